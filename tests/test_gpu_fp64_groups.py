"""The FP64 kernels' groups of 32 and 128 times, launch cuts and samples where they can go wrong.

Times around the group and chunk sizes, tiles of pvs that do not fill, sub-exposure counts beyond the offset
table, both Kepler paths and windows wider than a radian, times that are not finite; light curves within 1e-12
and gradients within 1e-10 (condition-scaled) of the FP64 oracle, and a pv's gradient the same bits however the
launch is cut.
"""
import numpy as np
import pytest

from oracle import grad as og
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


def check(rr, wl, grad_rows=2):
    import torch
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    f = m.evaluate(t, p, pb, wl.supersampling, wl.exptime)
    gbar = np.random.default_rng(3).normal(size=(wl.npv, wl.npt))
    g = m.evaluate_grad(t, p, torch.as_tensor(gbar, device=t.device), pb, wl.supersampling, wl.exptime).cpu().numpy()
    m.sync_status()
    s = om.build(wl.grid, wl.ld_model, wl.npb, wl.chromatic, wl.profiles, wl.n_general)
    ref = om.evaluate_workload(wl, s)
    assert np.abs(f.cpu().numpy() - ref).max() <= 1e-12
    for i in range(min(grad_rows, wl.npv)):
        J = og.jacobian(s, wl.times, wl.pb_index, wl.params[i], wl.supersampling, wl.exptime)
        scale = np.abs(gbar[i]) @ np.abs(J)
        err = np.abs(g[i] - gbar[i] @ J) / np.maximum(scale, max(1e-3 * scale.max(), 1e-300))
        assert err.max() < 1e-10
    return ref


@pytest.mark.parametrize("npv,npt", [(1, 1), (1, 31), (2, 33), (33, 127), (3, 128), (5, 129), (1, 1023), (40, 1025)])
def test_group_edges(rr, npv, npt):
    wl = W.make_small("quadratic", npv=npv, npt=npt, seed=npt, precision="fp64", span=0.02 * npt)
    check(rr, wl)


@pytest.mark.parametrize("ss", [(2,), (7, 1), (600, 3), (1024, 1024)])
def test_sub_exposures(rr, ss):
    wl = W.make_small("nonlinear", npv=2, npt=140, npb=len(ss), ss=ss, exptime=(0.03, 0.05), seed=8, precision="fp64", span=1.5)
    assert (check(rr, wl, 1) < 1).any()


@pytest.mark.parametrize("e,a", [(0.0, 2.0), (0.3, 2.3), (0.79, 12.0), (0.801, 12.0), (0.95, 60.0)])
def test_kepler_paths(rr, e, a):
    wl = W.make_small("quadratic", npv=7, npt=700, seed=4, precision="fp64", span=4.0)
    wl.params[:, 4] = e
    wl.params[:, 2] = a
    wl.params[:, 3] *= 0.3
    assert (check(rr, wl) < 1).any()


def test_times_that_are_not_finite(rr):
    """A time that is not finite gives 1 and changes nothing else, the first of a group included."""
    import torch
    wl = W.make_small("quadratic", npv=9, npt=900, seed=21, precision="fp64", span=3.0)
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    ref = m.evaluate(t, p, pb)
    bad = [0, 1, 32, 128, 255, 300, 899]
    t2 = t.clone()
    t2[bad] = torch.tensor([np.nan, np.inf, np.nan, np.nan, -np.inf, np.inf, np.nan], dtype=torch.float64, device=t.device)
    f = m.evaluate(t2, p, pb)
    keep = torch.ones(900, dtype=torch.bool, device=t.device)
    keep[bad] = False
    assert torch.equal(f[:, keep], ref[:, keep]) and bool((f[:, ~keep] == 1).all())


def test_gradient_does_not_depend_on_the_cut(rr):
    """A pv alone (per-group sums) and among 3,000 (chunk sums): the same bits."""
    import torch
    wl = W.make_small("quadratic", npv=3000, npt=9001, seed=2, precision="fp64", span=9.0)
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    gen = torch.Generator(device=t.device).manual_seed(1)
    gbar = torch.randn((3000, 9001), dtype=torch.float64, device=t.device, generator=gen)
    full = m.evaluate_grad(t, p, gbar, pb)
    for i in (0, 17, 2999):
        one = m.evaluate_grad(t, p[i:i + 1].contiguous(), gbar[i:i + 1].contiguous(), pb)
        assert torch.equal(one[0], full[i])
