"""GPU: the row passes of the double-float FFT that multiply by 1/Psi and pad or crop, and the band masks
of its column passes, against the same plan through the deconvolution passes and cuFFT Z2Z
(HVOX_DF_FFT=0): one grid and batches of several, both signs and directions, y columns in pairs and
single (n2y above 1,717), lengths with every radix.

Tolerance: the 1e-11 of the other comparisons with Z2Z (both transforms hold ~48 bits, amplified by
at most 1e2 in 1/Psi and 1/Phi at these upsamplings)."""
import numpy as np
import pytest
import torch

import oracle
from hvox_inputs import configs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius,cap,sigma,budget,isign", [(25.0, 10.0, 2.0, 1e9, -1), (170.0, 30.0, 2.0, 1e9, 1),
                                                           (400.0, 35.0, 2.0, 8e6, -1), (1500.0, 15.0, 1.5, 1e9, 1)])
def test_folded_passes_match_z2z(gpu_lib, monkeypatch, radius, cap, sigma, budget, isign):
    w = configs.small_case(seed=int(radius), n_pix=701, n_vis=907, cap_deg=cap, radius_m=radius)
    vis = configs.visibilities_cn(9, w.n_vis)
    out = []
    for own in ("1", "0"):
        monkeypatch.setenv("HVOX_DF_FFT", own)
        plan = gpu_lib.Plan(w.pix, w.uvw, 1e-9, isign=isign, mode="nufft", upsampfac=sigma, chunk_budget_bytes=budget)
        assert (plan.info()["fft_batches_df"] > 0) == (own == "1")
        V = plan.synthesize(torch.as_tensor(w.sky, dtype=torch.float64, device="cuda")).cpu().numpy()
        out.append((V, plan.analyze(torch.as_tensor(vis, dtype=torch.complex128, device="cuda")).cpu().numpy()))
        plan.close()
    assert max(oracle.rel_l2(a, b) for a, b in zip(*out)) <= 1e-11
