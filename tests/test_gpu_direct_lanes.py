"""The direct model's FP32 weight pass, four lanes per g node, where its tiling can go wrong.

Rows whose nodes do not fill a CTA, one-bin bands, the smallest grids, every count of bases per walk (1, 3,
5, 6 of a table), radius ratios from far below an annulus to almost the star's, and a radial grid whose
tables exceed the pass's shared memory (the thread-per-node pass).  Flux within the mixed form's 1e-6 of the
FP64 oracle.
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


def grid(nzin, nzlimb, ng, zcut=0.7):
    return dict(zcut=zcut, nzin=nzin, nzlimb=nzlimb, ng=ng, nk=60, k0=0.005, k1=0.3)


CASES = {
    "one-row": dict(npv=1, ng=200, nz=(200, 300), ld_model="quadratic"),
    "smallest-grid": dict(npv=5, ng=2, nz=(1, 1), ld_model="quadratic"),
    "few-annuli": dict(npv=7, ng=33, nz=(3, 2), ld_model="nonlinear", k_range=(0.3, 0.95)),
    "ragged-ng": dict(npv=19, ng=37, nz=(60, 90), ld_model="uniform"),
    "tiny-planets": dict(npv=6, ng=64, nz=(200, 300), ld_model="quadratic", k_range=(1e-4, 2e-3)),
    "giant-planets": dict(npv=6, ng=101, nz=(200, 300), ld_model="quadratic", k_range=(0.9, 0.99)),
    "two-walks": dict(npv=3, ng=50, nz=(40, 60), ld_model="tabulated", npb=9),
    "own-table": dict(npv=3, ng=50, nz=(40, 60), ld_model="tabulated", npb=3, chromatic=True),
    "largest-in-shared": dict(npv=2, ng=40, nz=(1400, 1000), ld_model="quadratic"),
    "beyond-shared": dict(npv=2, ng=40, nz=(2000, 2000), ld_model="quadratic"),
}


@pytest.mark.parametrize("name", CASES)
def test_direct_lanes_flux_matches_oracle(rr, name):
    import torch
    c = dict(CASES[name])
    ng, nz, npv = c.pop("ng"), c.pop("nz"), c.pop("npv")
    wl = W.make_small(npv=npv, npt=900, seed=61, span=6.0, direct=True, eccentric=True, **c)
    wl.grid = grid(*nz, ng)
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    f = m.evaluate(t, p, pb, wl.supersampling, wl.exptime).double().cpu().numpy()
    m.sync_status()
    s = om.build(wl.grid, wl.ld_model, wl.npb, wl.chromatic, wl.profiles, wl.n_general, direct=True)
    ref = om.evaluate_workload(wl, s)
    assert (ref < 1).any()
    assert np.abs(f - ref).max() <= 1e-6
    # the adjoint's layout holds the same rows: bitwise the same light curves
    ws = m.prepare(t, p, pb, wl.supersampling, wl.exptime)
    g = m.evaluate(t, p, pb, wl.supersampling, wl.exptime, prepared=ws).double().cpu().numpy()
    assert np.array_equal(f, g)
