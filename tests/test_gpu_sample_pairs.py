"""Sub-exposures evaluated two at a time: every sub-exposure count, candidate boundary and orbit path.

Odd and even counts, passbands of one sub-exposure between longer ones (pairs across two times), circular
and eccentric orbits up to the FP64 solve, and anomaly offsets beyond the series' range match the FP64 oracle
within the mixed form's 1e-6; the counting form, which takes one sample at a time, gives the same bits.
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


def check(rr, wl):
    import torch
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    f = m.evaluate(t, p, pb, wl.supersampling, wl.exptime)
    m.count_samples(True)
    g = m.evaluate(t, p, pb, wl.supersampling, wl.exptime)
    m.count_samples(False)
    m.sync_status()
    assert torch.equal(f, g)
    ref = om.evaluate_workload(wl, om.build(wl.grid, wl.ld_model, wl.npb, wl.chromatic, wl.profiles, wl.n_general))
    assert (ref < 1).mean() > 0.01 and np.abs(f.double().cpu().numpy() - ref).max() <= 1e-6


@pytest.mark.parametrize("ss", [(2,), (3,), (31,), (7, 1), (1, 30, 2), (1, 1, 5, 10)])
def test_counts(rr, ss):
    check(rr, W.make_small("nonlinear", npv=5, npt=901, npb=len(ss), ss=ss, exptime=(0.02,) * len(ss), seed=3, span=2.0))


@pytest.mark.parametrize("e,a", [(0.0, 12.0), (0.0, 1.3), (0.3, 2.3), (0.79, 12.0), (0.81, 12.0)])
def test_orbits(rr, e, a):
    wl = W.make_small("quadratic", npv=7, npt=700, npb=2, ss=(1, 4), exptime=(0.0, 0.03), seed=4, span=4.0)
    wl.params[:, 4], wl.params[:, 2] = e, a
    wl.params[:, 3] *= 0.3
    check(rr, wl)
