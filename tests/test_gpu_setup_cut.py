"""The set-up launch's kinds of CTAs and row widths where they can go wrong.

Numbers of pvs around a header CTA's and a row CTA's share, 1 to 32 passbands, g grids whose rows are and are not
16-byte aligned, every model and both layouts: light curves against the FP64 oracle (1e-12 FP64, 1e-6 mixed),
the status words of invalid pvs at the edges exactly, and a pv alone bitwise what it is in the batch.
"""
import numpy as np
import pytest

from oracle import model as om
from paper_2009_08500_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "mixed": 1e-6}


@pytest.fixture(scope="module")
def rr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2009_08500_gb300 import rr as _rr
    _rr.load_library()
    return _rr


CASES = [
    dict(ld_model="quadratic", npv=31, ng=200), dict(ld_model="quadratic_tri", npv=33, ng=198),
    dict(ld_model="nonlinear", npv=65, ng=199), dict(ld_model="nonlinear", npv=5, ng=201, npb=2, chromatic=True),
    dict(ld_model="tabulated", npv=9, ng=200, npb=9), dict(ld_model="quadratic", npv=3, ng=37, npb=32, chromatic=True),
    dict(ld_model="uniform", npv=40, ng=2), dict(ld_model="quadratic", npv=17, ng=50, npb=3, direct=True, chromatic=True),
    dict(ld_model="quadratic", npv=17, ng=52, npb=3, direct=True, chromatic=True, shared_weights=True),
    dict(ld_model="linear", npv=34, ng=61, direct=True),
]


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: f"{c['ld_model']}-{c['npv']}-ng{c['ng']}-pb{c.get('npb', 1)}-d{int(c.get('direct', 0))}")
def test_setup_cut(rr, case, precision):
    import torch
    c = dict(case)
    ng = c.pop("ng")
    wl = W.make_small(npt=331, seed=17, precision=precision, span=4.0, **c)
    wl.grid = dict(wl.grid, ng=ng)
    bad = sorted({0, wl.npv // 2})
    wl.params[bad[0], 1] = -1.0
    wl.params[bad[-1], 4] = np.nan
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    st = torch.full((wl.npv,), -1, dtype=torch.int32, device=t.device)
    f = m.evaluate(t, p, pb, wl.supersampling, wl.exptime, pv_status=st)
    s = om.build(wl.grid, wl.ld_model, wl.npb, wl.chromatic, wl.profiles, wl.n_general, direct=wl.direct,
                 shared=wl.shared_weights)
    ref, rst = om.evaluate_workload(wl, s, return_status=True)
    assert np.array_equal(st.cpu().numpy(), rst) and rst[bad].all()
    ok = rst == 0
    if ok.any():
        assert np.abs(f.cpu().numpy()[ok] - ref[ok]).max() <= TOL[precision]
    assert bool(torch.isnan(f[torch.as_tensor(~ok)]).all())
    if m.nparam > 64:
        return
    g = torch.randn(f.shape, dtype=f.dtype, device=f.device, generator=torch.Generator(device=f.device).manual_seed(1))
    ws = m.prepare(t, p, pb, wl.supersampling, wl.exptime)
    fb, gb = m.evaluate_both(t, p, g, ws, pb, wl.supersampling, wl.exptime)
    assert torch.equal(fb.nan_to_num(nan=-1.0), f.nan_to_num(nan=-1.0))
    for i in (1, wl.npv - 1):
        one = m.evaluate_grad(t, p[i:i + 1].contiguous(), g[i:i + 1].contiguous(), pb, wl.supersampling, wl.exptime)
        assert torch.equal(one[0].nan_to_num(nan=-1.0), gb[i].nan_to_num(nan=-1.0))
        f1 = m.evaluate(t, p[i:i + 1].contiguous(), pb, wl.supersampling, wl.exptime)
        assert torch.equal(f1[0].nan_to_num(nan=-1.0), f[i].nan_to_num(nan=-1.0))
