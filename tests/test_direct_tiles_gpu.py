"""GPU: the tensor-core direct sums at the edges of their tiles (256 owners, 128 streamed
points, chunks of 64 or 32 columns, segments from 64 points) and at the edges of their
coordinate range, against the FP64 oracle.

Tolerances. FP32: the hardware sine's error (2^-20.9) and the phase's (2 pi 7e-8) bound a term's
error by 1.1e-6, and 10 eps = 1e-5 leaves room for cancellation in the sums. Double-float: a
term's error is below 5e-10 per part (the table entry's low part rotated in FP32), 1e-9 for
the sums. Coordinates kept as float pairs round a product of t turns by t 2^-48 in each of two
factors, so a case of t turns per dimension adds 2 pi 3 t 2^-47."""
import math

import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


def _points(n_pix, n_vis, radius, pix_scale=1.0, seed=0):
    rng = np.random.default_rng([n_pix, n_vis, seed])
    xy = rng.uniform(-0.5, 0.5, (n_pix, 2))
    pix = np.concatenate([xy, np.sqrt(1.0 - (xy * xy).sum(1))[:, None]], axis=1) * pix_scale
    uvw = rng.uniform(-radius, radius, (n_vis, 3)) / pix_scale
    sky = rng.lognormal(0.0, 1.0, n_pix)
    vis = rng.normal(size=n_vis) + 1j * rng.normal(size=n_vis)
    return pix, uvw, sky, vis


def _check(hv, eps, pix, uvw, sky, vis, isign, tol):
    plan = hv.Plan(pix, uvw, eps, isign=isign, mode="direct")
    V = plan.synthesize(torch.as_tensor(sky, dtype=plan.real_dtype, device="cuda"))
    I = plan.analyze(torch.as_tensor(vis, dtype=plan.complex_dtype, device="cuda"))
    plan.sync()
    plan.close()
    e_v = oracle.rel_l2(V.cpu().numpy(), oracle.sky2vis(pix, uvw, sky, isign=isign))
    e_i = oracle.rel_l2(I.cpu().numpy(), oracle.vis2sky(pix, uvw, vis, isign=isign))
    print(f"eps {eps:g} {len(pix)} x {len(uvw)}: {e_v:.2e} {e_i:.2e}")
    assert e_v <= tol and e_i <= tol, (e_v, e_i)


@pytest.mark.parametrize("eps", [1e-6, 1e-9])
@pytest.mark.parametrize("n_pix,n_vis", [(1, 1), (63, 255), (64, 256), (65, 257), (127, 33), (128, 128), (129, 511),
                                         (2048, 2049), (2113, 700), (300, 6000)])
def test_tile_edges(gpu_lib, eps, n_pix, n_vis):
    tol = 1e-5 if eps == 1e-6 else 1e-9
    _check(gpu_lib, eps, *_points(n_pix, n_vis, 3e4), -1 if n_pix % 2 else 1, tol)


# radius * pix_scale is the turns per dimension: inside the digits' reach of either form, at the
# reach of the FP32 form (2^28) and past it (the double-float form on float values), and past
# the double-float reach (2^33: FP64 kernels); coordinates far from unit size.
@pytest.mark.parametrize("eps,radius,scale", [(1e-6, 2.0 ** 22, 1.0), (1e-4, 0.9 * 2.0 ** 28, 1.0),
                                              (1e-4, 1.5 * 2.0 ** 28, 1.0), (1e-9, 2.0 ** 20, 1.0),
                                              (1e-6, 1e3, 1e3), (1e-6, 1e3, 1e-7), (1e-9, 1e3, 3e5), (1e-9, 1e3, 1e-5),
                                              (1e-9, 1.5 * 2.0 ** 33, 1.0)])
def test_coordinate_range(gpu_lib, eps, radius, scale):
    split = 0.0 if radius > 2.0 ** 33 else 2.0 * math.pi * 3.0 * radius * 2.0 ** -47
    fp64 = 2.0 * math.pi * 3.0 * radius * 2.0 ** -52 if radius > 2.0 ** 33 else 0.0  # plain FP64 products
    tol = (1e-9 if eps == 1e-9 else 1e-5) + split + fp64
    _check(gpu_lib, eps, *_points(300, 700, radius, scale), -1, tol)


@pytest.mark.parametrize("n_pix,n_vis,radius", [(1, 1, 1e3), (65, 257, 3e4), (300, 1000, 1.5 * 2.0 ** 28)])
def test_noalloc_edges(gpu_lib, n_pix, n_vis, radius):
    pix, uvw, sky, _ = _points(n_pix, n_vis, radius)
    V = torch.empty(n_vis, dtype=torch.complex64, device="cuda")
    gpu_lib.direct_synthesize_noalloc(torch.as_tensor(pix, device="cuda"), torch.as_tensor(uvw, device="cuda"),
                                      torch.as_tensor(sky, dtype=torch.float32, device="cuda"), V, isign=1)
    torch.cuda.synchronize()
    tol = 1e-5 + 2.0 * math.pi * 3.0 * radius * 2.0 ** -47
    assert oracle.rel_l2(V.cpu().numpy(), oracle.sky2vis(pix, uvw, sky, isign=1)) <= tol
