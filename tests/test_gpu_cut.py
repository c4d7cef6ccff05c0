"""Launches cut for few parameter vectors: light curves and gradients do not depend on the cut.

A pv alone, among 40 and among 2,500 (an uncut launch) gives the same bits, with one and with several
passbands and sub-exposures, for lengths that leave partial groups and chunks; and the cut launches of
vectors that all transit together match the FP64 oracle within the mixed form's 1e-6.
"""
import numpy as np
import pytest

from oracle import model as om
from paper_2009_08500_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2009_08500_gb300 import rr as _rr
    _rr.load_library()
    return _rr


def ensemble(npv, npt, **kw):
    """Vectors scattered about one planet, times about its transits."""
    wl = W.make_small(npv=npv, npt=npt, seed=5, **kw)
    rng = np.random.default_rng(1)
    wl.params[:] = wl.params[0] * (1.0 + 1e-3 * rng.standard_normal(wl.params.shape))
    T0, P = wl.params[0, 0], wl.params[0, 1]
    wl.params[:, 0], wl.params[:, 1] = T0 + 1e-4 * rng.standard_normal(npv), P
    wl.times = np.sort(T0 + P * rng.integers(0, 4, npt) + 0.2 * P * rng.uniform(-1, 1, npt))
    return wl


CASES = [dict(ld_model="quadratic", npt=9001), dict(ld_model="quadratic_tri", npt=1023, ss=(7,), exptime=(0.02,)),
         dict(ld_model="nonlinear", npt=4100, npb=3, chromatic=True, ss=(1, 4, 9), exptime=(0.0, 0.01, 0.02)),
         dict(ld_model="tabulated", npt=2050, npb=4)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c['ld_model']}-{c['npt']}")
def test_results_do_not_depend_on_the_cut(rr, case):
    import torch
    wl = ensemble(2500, **case)
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    ss, ex = wl.supersampling, wl.exptime
    g = torch.randn((wl.npv, wl.npt), device=t.device, generator=torch.Generator(device=t.device).manual_seed(2))
    f = m.evaluate(t, p, pb, ss, ex)
    full = m.evaluate_grad(t, p, g, pb, ss, ex)
    for lo, n in ((0, 1), (1237, 1), (2460, 40), (100, 9)):
        q, gq = p[lo:lo + n].contiguous(), g[lo:lo + n].contiguous()
        assert torch.equal(m.evaluate(t, q, pb, ss, ex), f[lo:lo + n])
        assert torch.equal(m.evaluate_grad(t, q, gq, pb, ss, ex), full[lo:lo + n])
        ws = m.prepare(t, q, pb, ss, ex)
        fb, gb = m.evaluate_both(t, q, gq, ws, pb, ss, ex)
        assert torch.equal(fb, f[lo:lo + n]) and torch.equal(gb, full[lo:lo + n])
    m.sync_status()


@pytest.mark.parametrize("npv,npt", [(1, 129), (3, 1024), (8, 257), (9, 2049), (31, 640)])
def test_cut_launch_matches_oracle(rr, npv, npt):
    wl = ensemble(npv, npt, ld_model="quadratic", npb=2, ss=(1, 3), exptime=(0.0, 0.01))
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    f = m.evaluate(t, p, pb, wl.supersampling, wl.exptime).double().cpu().numpy()
    ref = om.evaluate_workload(wl, om.build(wl.grid, wl.ld_model, wl.npb, wl.chromatic, wl.profiles, wl.n_general))
    assert (ref < 1).mean() > 0.05 and np.abs(f - ref).max() <= 1e-6
