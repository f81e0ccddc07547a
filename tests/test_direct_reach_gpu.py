"""GPU: direct sums of FP32 plans (and of the call that allocates nothing) at eps = 1e-6 over the reach of
their digits, 2^28 turns per dimension.

Tolerance: 2e-6 for the hardware sine (2^-20.9 a term) and the FP32 sums, as at small phases, plus
what float pairs cost: a coordinate kept as hi + lo is off by at most 2^-49 of itself, uniformly, so a
product of t turns by at most sqrt(2) 2^-49 t / sqrt(3) rms and three of them by 2 pi sqrt(2) 2^-49 t
radians. Nothing for the digits."""
import math

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _points(n_pix, n_vis, radius, scale=1.0):
    rng = np.random.default_rng([n_pix, n_vis])
    xy = rng.uniform(-0.5, 0.5, (n_pix, 2))
    pix = np.concatenate([xy, np.sqrt(1.0 - (xy * xy).sum(1))[:, None]], axis=1) * scale
    uvw = rng.uniform(-radius, radius, (n_vis, 3)) / scale
    return pix, uvw, rng.lognormal(0.0, 1.0, n_pix), rng.normal(size=n_vis) + 1j * rng.normal(size=n_vis)


def _errors(hv, eps, pix, uvw, sky, vis):
    plan = hv.Plan(pix, uvw, eps, precision="fp32", mode="direct")
    V = plan.synthesize(torch.as_tensor(sky, dtype=torch.float32, device="cuda"))
    I = plan.analyze(torch.as_tensor(vis, dtype=torch.complex64, device="cuda"))
    plan.sync()
    plan.close()
    Va = torch.empty(len(uvw), dtype=torch.complex64, device="cuda")
    hv.direct_synthesize_noalloc(torch.as_tensor(pix, device="cuda"), torch.as_tensor(uvw, device="cuda"),
                                 torch.as_tensor(sky, dtype=torch.float32, device="cuda"), Va)
    ref = oracle.sky2vis(pix, uvw, sky)
    return [oracle.rel_l2(V.cpu().numpy(), ref), oracle.rel_l2(I.cpu().numpy(), oracle.vis2sky(pix, uvw, vis)),
            oracle.rel_l2(Va.cpu().numpy(), ref)]


@pytest.mark.parametrize("scale", [1.0, 3e4])
@pytest.mark.parametrize("log2", [20, 22, 24, 26, 27, 27.8])
def test_fp32_digits_hold_over_their_reach(gpu_lib, log2, scale):
    radius = 2.0 ** log2
    e = _errors(gpu_lib, 1e-6, *_points(400, 900, radius, scale))
    print(f"2^{log2}: {e}")
    assert max(e) <= 2e-6 + 2.0 * math.pi * math.sqrt(2.0) * radius * 2.0 ** -49


# Past the double-float digits (2^33 turns; their leading one is inexact in fp16 from 2^34 and infinite from
# 2^39) the sums run in FP64, as the oracle's: a product of t turns rounds at 2^-53 t in each. Baselines within
# 2e3 wavelengths of a far point: the host sizes grids by extents, slowly where these are 2^36.
@pytest.mark.parametrize("log2", [33.5, 36, 40])
def test_sums_beyond_every_digit(gpu_lib, log2):
    pix, uvw, sky, vis = _points(400, 900, 1e3)
    uvw += 2.0 ** log2 * np.array([1.0, -1.0, 1.0])
    e = _errors(gpu_lib, 1e-4, pix, uvw, sky, vis)
    print(f"2^{log2}: {e}")
    assert max(e) <= 1e-6 + 2.0 * math.pi * 3.0 * 2.0 ** log2 * 2.0 ** -52
