"""FP64 light curves written by the adjoint kernel: the bits of the separate calls.

Odd and even lengths, partial groups, several passbands and passband indices out of range, per-passband radius
ratios, shared direct weights, zero cotangents (one time, most times, whole vectors), invalid vectors, both
Kepler paths, one vector and many.
"""
import numpy as np
import pytest

from paper_2009_08500_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2009_08500_gb300 import rr as _rr
    _rr.load_library()
    return _rr


CASES = [dict(npv=1, npt=129), dict(npv=1, npt=2000), dict(npv=67, npt=1023), dict(npv=700, npt=3000),
         dict(npv=33, npt=500, npb=3, chromatic=True), dict(npv=9, npt=770, npb=4, ld_model="nonlinear"),
         dict(npv=20, npt=640, npb=2, chromatic=True, direct=True, shared_weights=True),
         dict(npv=12, npt=515, e=0.81, a=12.0), dict(npv=12, npt=515, eccentric=False)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(str(v) for v in c.values()))
def test_both_equals_separate_calls(rr, case):
    import torch
    case = dict(case)
    e, a = case.pop("e", None), case.pop("a", None)
    wl = W.make_small(**{"ld_model": "quadratic", **case}, seed=11, precision="fp64", span=5.0)
    if e is not None:
        wl.params[:, 4], wl.params[:, 2] = e, a
        wl.params[:, 3] *= 0.3
    if wl.npv > 8:
        wl.params[5, 1] = -1.0   # an invalid vector
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    if pb is not None and wl.npb > 1:
        pb[[0, 200, wl.npt - 1]] = wl.npb + 3
    gen = torch.Generator(device=t.device).manual_seed(1)
    g = torch.randn((wl.npv, wl.npt), dtype=torch.float64, device=t.device, generator=gen)
    zeros = g.clone()
    zeros[:, ::3] = 0.0
    zeros[wl.npv // 2:, : wl.npt // 2] = 0.0
    for gbar in (g, zeros, torch.zeros_like(g)):
        f, gr = m.evaluate(t, p, pb), m.evaluate_grad(t, p, gbar, pb)
        ws = m.prepare(t, p, pb)
        fb, gb = m.evaluate_both(t, p, gbar, ws, pb)
        m.sync_status()
        assert torch.equal(fb.isnan(), f.isnan()) and torch.equal(fb.nan_to_num(), f.nan_to_num())
        assert torch.equal(gb.isnan(), gr.isnan()) and torch.equal(gb.nan_to_num(), gr.nan_to_num())
    assert wl.npt < 130 or bool((f < 1).any())
