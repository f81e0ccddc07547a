"""GPU: the mean error of the FP32 direct sums' cosine over a turn. A sum of N positive values multiplies it by N while
the sum itself grows as sqrt(N), so it is the error of long baselines' visibilities over large skies.

2^20 pixels with log-normal values, 64 long baselines, against FP64. Bounds: 3e-6 for the visibilities (with 2 pi
rounded to float in every column the mean of 1.2e-8 makes 7.6e-6 of them; sines, phases, sums and what is left of
the mean 1e-6); the mean itself, Re(V - exact) / sum(c) over the baselines, 1.3e-9: half of the 2.3e-9 by which
one column in 32 with the other factor moves it, and rounding (1e-6 |V| / sum(c) / sqrt(64) = 2e-10)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def test_positive_sums_on_long_baselines(gpu_lib):
    rng = np.random.default_rng(2306)
    n_pix, n_vis = 1 << 20, 64
    xy = rng.uniform(-0.5, 0.5, (n_pix, 2))
    pix = np.concatenate([xy, np.sqrt(1.0 - (xy * xy).sum(1))[:, None]], axis=1)
    uvw = rng.uniform(-3e4, 3e4, (n_vis, 3))
    sky = rng.lognormal(0.0, 1.0, n_pix).astype(np.float32)
    plan = gpu_lib.Plan(pix, uvw, 1e-6, precision="fp32", mode="direct")
    V = plan.synthesize(torch.as_tensor(sky, device="cuda")).cpu().numpy().astype(np.complex128)
    plan.close()
    ref = oracle.sky2vis(pix, uvw, sky.astype(np.float64))
    mean = float((V - ref).real.mean() / sky.sum(dtype=np.float64))
    err = oracle.rel_l2(V, ref)
    print(f"rel_l2 {err:.2e}, mean error of the cosine {mean:.2e}")
    assert err <= 3e-6 and abs(mean) <= 1.3e-9
