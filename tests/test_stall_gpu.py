"""GPU: the direct kernels' bounded waits run out. The producers of a stalled launch keep their tiles to
themselves (HVOX_FAULT=stall:n, read on the host), so that every wait behind them ends at its limit
with nothing in flight on the tensor cores: the call reports HVOX_ETIMEOUT, every output that misses
terms is NaN, none is finite and short, and the context stays usable."""
import time

import numpy as np
import pytest
import torch

import oracle
from hvox_inputs import configs

pytestmark = pytest.mark.gpu


@pytest.fixture
def stalled(monkeypatch):
    def make(call):
        monkeypatch.setenv("HVOX_FAULT", "stall:1")
        try:
            return call()
        finally:
            monkeypatch.delenv("HVOX_FAULT")
    return make


def _finite_rows_match(V, ref, tol):
    ok = np.isfinite(V)
    if ok.any():
        assert np.abs(V[ok] - ref[ok]).max() <= tol * np.abs(ref).max()
    return ok


def _clean_plan(gpu_lib, w, eps):
    plan = gpu_lib.Plan(w.pix, w.uvw, eps, mode="direct")
    V = plan.synthesize(torch.as_tensor(w.sky, dtype=plan.real_dtype, device="cuda")).cpu().numpy()
    plan.close()
    assert oracle.rel_l2(V, oracle.sky2vis(w.pix, w.uvw, w.sky)) <= 1e-5


# more owner tiles x segments than CTAs (items taken after the stalled one), and a single item
@pytest.mark.parametrize("eps,n_pix,n_vis", [(1e-6, 40, 90), (1e-6, 3001, 60000), (1e-9, 3001, 60000)])
def test_stalled_plan_reports_timeout(gpu_lib, stalled, eps, n_pix, n_vis):
    w = configs.small_case(seed=31, n_pix=n_pix, n_vis=n_vis)
    plan = stalled(lambda: gpu_lib.Plan(w.pix, w.uvw, eps, mode="direct"))
    sky = torch.as_tensor(w.sky, dtype=plan.real_dtype, device="cuda")
    vis = torch.ones(n_vis, dtype=plan.complex_dtype, device="cuda")
    for call, arg in ((plan.synthesize, sky), (plan.analyze, vis)):
        torch.cuda.synchronize()
        t0 = time.monotonic()
        out = call(arg)
        torch.cuda.synchronize()
        took = time.monotonic() - t0
        print(f"eps {eps:g} {n_pix} x {n_vis}: {took:.2f} s")
        assert took < 30.0
        with pytest.raises(gpu_lib.HvoxError) as e:
            plan.sync()
        assert e.value.code == 4  # HVOX_ETIMEOUT
        plan.sync()  # the report cleared the word
        assert not torch.isfinite(torch.view_as_real(out) if out.is_complex() else out).any()
    plan.close()
    _clean_plan(gpu_lib, w, eps)


def test_stalled_plan_in_a_batch_leaves_no_short_sums(gpu_lib, stalled):
    w = configs.small_case(seed=32, n_pix=2001, n_vis=30000)
    u = configs.small_case(seed=33, n_pix=1501, n_vis=25000)
    bad = stalled(lambda: gpu_lib.Plan(w.pix, w.uvw, 1e-6, mode="direct"))
    good = gpu_lib.Plan(u.pix, u.uvw, 1e-6, mode="direct")
    ins = [torch.as_tensor(x.sky, dtype=torch.float32, device="cuda") for x in (w, u)]
    V = [v.cpu().numpy() for v in gpu_lib.synthesize_batch([bad, good], ins)]
    with pytest.raises(gpu_lib.HvoxError) as e:
        bad.sync()
    assert e.value.code == 4
    assert not np.isfinite(V[0]).any()
    ref = oracle.sky2vis(u.pix, u.uvw, u.sky)
    ok = _finite_rows_match(V[1], ref, 1e-4)
    if ok.all():
        good.sync()
    else:
        with pytest.raises(gpu_lib.HvoxError) as e:
            good.sync()
        assert e.value.code == 4
    bad.close()
    good.close()
    _clean_plan(gpu_lib, u, 1e-6)


def test_stalled_noalloc_call_is_nan(gpu_lib, stalled):
    # more items than CTAs: those that a stopped CTA had left were missing from finite sums
    w = configs.small_case(seed=34, n_pix=3001, n_vis=60000)
    pix = torch.as_tensor(w.pix, device="cuda")
    uvw = torch.as_tensor(w.uvw, device="cuda")
    sky = torch.as_tensor(w.sky, dtype=torch.float32, device="cuda")
    V = torch.zeros(w.n_vis, dtype=torch.complex64, device="cuda")
    stalled(lambda: gpu_lib.direct_synthesize_noalloc(pix, uvw, sky, V))
    torch.cuda.synchronize()
    assert not torch.isfinite(torch.view_as_real(V)).any()
    gpu_lib.direct_synthesize_noalloc(pix, uvw, sky, V)
    torch.cuda.synchronize()
    assert oracle.rel_l2(V.cpu().numpy(), oracle.sky2vis(w.pix, w.uvw, w.sky)) <= 1e-5
