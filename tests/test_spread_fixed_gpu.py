"""GPU: spreading of FP64 plans into fixed-point tiles at the edges of its rules: every kernel width
of the range, bins that share one tile, bins swept in slabs of planes (deep windows over a
dense patch), bins split into runs, and groups too wide for a tile (added straight to the
grid), against the FP64 oracle.

Tolerance: 10 eps, the bound of the other FP64 NUFFT tests, down to the 1e-9 of the double-float
arithmetic."""
import numpy as np
import pytest
import torch

import oracle
from hvox_inputs import configs

pytestmark = pytest.mark.gpu


# radius and cap (with the fixed point counts) set the points per grid cell, hence the extent of a bin of 128
# points; eps and upsampling the kernel width (9 to 16)
@pytest.mark.parametrize("eps,sigma", [(3e-7, 2.0), (1e-8, 2.0), (1e-9, 2.0), (1e-9, 1.5), (1e-9, 1.25)])
@pytest.mark.parametrize("radius,cap", [(20.0, 20.0), (120.0, 20.0), (120.0, 60.0), (500.0, 35.0)])
def test_fixed_tile_spreading(gpu_lib, eps, sigma, radius, cap):
    w = configs.small_case(seed=int(radius + cap), n_pix=1501, n_vis=1607, cap_deg=cap, radius_m=radius)
    plan = gpu_lib.Plan(w.pix, w.uvw, eps, mode="nufft", upsampfac=sigma)
    vis = configs.visibilities_cn(3, w.n_vis)
    V = plan.synthesize(torch.as_tensor(w.sky, dtype=torch.float64, device="cuda")).cpu().numpy()
    I = plan.analyze(torch.as_tensor(vis, dtype=torch.complex128, device="cuda")).cpu().numpy()
    plan.close()
    assert oracle.rel_l2(V, oracle.sky2vis(w.pix, w.uvw, w.sky)) <= 10 * max(eps, 1e-9)
    assert oracle.rel_l2(I, oracle.vis2sky(w.pix, w.uvw, vis)) <= 10 * max(eps, 1e-9)
