"""GPU: the FP32 FFT of NUFFT grids (with its folded deconvolution) against the same plan's grids
through the deconvolution passes and cuFFT C2C (HVOX_C_FFT=0), and against the FP64 oracle:
one transform and a batch of several grids, radices 2 to 16, both signs and both directions.

Tolerance against cuFFT: both round each of ~log2(cells) <= 30 levels at 2^-24 of the data's
norm, and the grids' edges are amplified by at most 1e2 in 1/Psi and 1/Phi at these
upsamplings (2 and 1.5): 1e-5 in all, the FP32 bound of the other tests."""
import numpy as np
import pytest
import torch

import oracle
from hvox_inputs import configs

pytestmark = pytest.mark.gpu


def _both(gpu_lib, w, isign, **kw):
    plan = gpu_lib.Plan(w.pix, w.uvw, 1e-6, isign=isign, mode="nufft", **kw)
    vis = configs.visibilities_cn(9, w.n_vis)
    V = plan.synthesize(torch.as_tensor(w.sky, dtype=torch.float32, device="cuda")).cpu().numpy()
    I = plan.analyze(torch.as_tensor(vis, dtype=torch.complex64, device="cuda")).cpu().numpy()
    plan.profile("serial")
    plan.synthesize(torch.as_tensor(w.sky, dtype=torch.float32, device="cuda"))
    launches = plan.stats()["launches"]
    blocks = plan.info()["n_nufft_blocks"]
    plan.close()
    return V, I, launches, blocks


# radius and cap choose the grid lengths (radices 2 .. 16 among them); budgets below the whole grid give batches
@pytest.mark.parametrize("radius,cap,sigma,budget,isign", [(30.0, 10.0, 2.0, 1e9, -1), (100.0, 35.0, 1.5, 1e9, 1),
                                                           (170.0, 30.0, 2.0, 1e9, -1), (233.0, 35.0, 1.5, 2e6, 1),
                                                           (400.0, 35.0, 2.0, 4e6, -1), (1500.0, 20.0, 1.5, 1e9, 1)])
def test_fp32_fft_matches_cufft_and_oracle(gpu_lib, monkeypatch, radius, cap, sigma, budget, isign):
    covered = radius < 1500  # its y length, 4374 = 15 * 15 * ..., takes more than the 1024 threads of a CTA: cuFFT
    w = configs.small_case(seed=int(radius), n_pix=901, n_vis=1207, cap_deg=cap, radius_m=radius)
    kw = dict(upsampfac=sigma, chunk_budget_bytes=budget)
    V, I, own, blocks = _both(gpu_lib, w, isign, **kw)
    monkeypatch.setenv("HVOX_C_FFT", "0")
    Vc, Ic, ref, _ = _both(gpu_lib, w, isign, **kw)
    assert (own["deconv"] == 0) == covered and ref["deconv"] > 0, "the FP32 FFT did not run where it applies"
    e = [oracle.rel_l2(V, Vc), oracle.rel_l2(I, Ic)]
    vis = configs.visibilities_cn(9, w.n_vis)
    o = [oracle.rel_l2(V, oracle.sky2vis(w.pix, w.uvw, w.sky, isign=isign)),
         oracle.rel_l2(I, oracle.vis2sky(w.pix, w.uvw, vis, isign=isign))]
    print(f"radius {radius:g} cap {cap:g} sigma {sigma:g}: {blocks} sub-problems, vs cuFFT {e}, vs oracle {o}")
    assert max(e) <= 1e-5 and max(o) <= 1e-5
