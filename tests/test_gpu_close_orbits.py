"""Light curves of eccentric planets that pass close by the star, where Kepler's equation is solved far from conjunction.

a (1 - e) of 1.2 to 1.45 with e of 0.45 to 0.78: transit windows of a radian and more in mean anomaly, on one side of
the transit through periastron.  The mixed form's light curves (one and several samples per time) are finite and valid
for every vector, and within the mixed form's 1e-6 of the FP64 oracle.
"""
import numpy as np
import pytest

from oracle import model as om
from paper_2009_08500_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ss,ex", [((5,), (0.02,)), ((1,), (0.0,)), ((4, 1), (0.03, 0.0))])
def test_close_eccentric_orbits(ss, ex):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2009_08500_gb300 import rr
    wl = W.make_small("quadratic", npv=256, npt=5000, npb=len(ss), ss=ss, exptime=ex)
    wl.times = np.sort(np.random.default_rng(5).uniform(0.0, 27.5, wl.npt))
    rng = np.random.default_rng(9)
    p = wl.params
    p[:, 4] = rng.uniform(0.45, 0.78, wl.npv)
    p[:, 2] = rng.uniform(1.2, 1.45, wl.npv) / (1.0 - p[:, 4])
    p[:, 3] *= 0.1
    p[:, 6] = 0.1
    m = rr.model_for(wl)
    t, pb, dp = rr.to_device(wl)
    status = torch.empty(wl.npv, dtype=torch.int32, device=t.device)
    f = m.evaluate(t, dp, pb, wl.supersampling, wl.exptime, pv_status=status).double().cpu().numpy()
    m.sync_status()
    assert not status.any() and np.isfinite(f).all()
    rows = slice(0, 64)
    wl.params = p[rows]
    ref = om.evaluate_workload(wl, om.build(wl.grid, wl.ld_model, wl.npb, wl.chromatic, wl.profiles, wl.n_general))
    assert (ref < 1).mean() > 0.05 and np.abs(f[rows] - ref).max() <= 1e-6


def test_no_transit_is_lost_on_an_extreme_orbit():
    """A planet whose orbit crosses the star (a = 1.137, e = 0.747, k = 0.807): a solve that runs off to infinity must not
    pass for a planet out of transit.  FP32: 7e-7 in x, times a (1 + e) = 2 in z, times a slope of 0.8, some 1e-6; 5e-6."""
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2009_08500_gb300 import rr
    wl = W.make_small("quadratic", npv=8, npt=3000, seed=3, direct=True)
    p = wl.params
    p[:, :7] = [0.87076078, 2.29136833, 1.13654818, 1.07053115, 0.74653325, 5.31471914, 0.80711502]
    p[:, 5] += 0.02 * np.arange(8)
    wl.times = np.sort(np.random.default_rng(4).uniform(0.0, 300.0, wl.npt))
    m = rr.model_for(wl)
    t, pb, dp = rr.to_device(wl)
    f = m.evaluate(t, dp, pb).double().cpu().numpy()
    m.sync_status()
    ref = om.evaluate_workload(wl, om.build(wl.grid, wl.ld_model, wl.npb, wl.chromatic, wl.profiles, direct=True))
    assert (ref < 1).mean() > 0.05 and np.abs(f - ref).max() <= 5e-6
