"""The FP64 kernels' transit decisions (made in FP32 from a group's reference time) miss no transit.

Times 10^12 periods from T0 give the bits of the same phases near T0, and a group whose first time is a huge value (a fill
value, beyond FP32's range or not) gives its other times the bits they have without it.
"""
from fractions import Fraction

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


def test_times_many_periods_from_t0(rr):
    import torch
    wl = W.make_small("quadratic", npv=40, npt=1500, seed=3, precision="fp64")
    P = 1.0717e-3
    wl.params[:, 0], wl.params[:, 1] = 0.0, P
    wl.params[:, 3] *= 0.2
    wl.times = np.sort(1e9 + np.random.default_rng(1).uniform(0.0, 1.0, wl.npt))
    n = np.rint(wl.times * (1.0 / P))
    tau = np.array([float(Fraction(t) - int(k) * Fraction(P)) for t, k in zip(wl.times, n)])
    m = rr.model_for(wl)
    t, _, p = rr.to_device(wl)
    near = torch.as_tensor(tau, device=t.device)
    f, ref = m.evaluate(t, p), m.evaluate(near, p)
    assert bool((ref < 1).any()) and torch.equal(f, ref)
    g = torch.randn(f.shape, dtype=torch.float64, device=t.device, generator=torch.Generator(device=t.device).manual_seed(2))
    ga, gb = m.evaluate_grad(t, p, g), m.evaluate_grad(near, p, g)
    keep = [0, 2, 3, 4, 5, 6, 7, 8]   # (the period's derivative grows with the number of periods)
    scale = gb.abs().amax(0)
    assert bool(((ga - gb).abs()[:, keep] <= 1e-12 * scale[keep]).all())
    m.sync_status()


def test_huge_times(rr):
    import torch
    wl = W.make_small("quadratic", npv=40, npt=1500, seed=4, precision="fp64", span=3.0)
    m = rr.model_for(wl)
    t, _, p = rr.to_device(wl)
    bad = [0, 128, 129, 256, 512, 640, 777]
    t2 = t.clone()
    t2[bad] = torch.tensor([1.7e308, -1e300, 1e300, 1e39, -3e38, 1e30, 1.7e308], dtype=torch.float64, device=t.device)
    g = torch.randn((wl.npv, wl.npt), dtype=torch.float64, device=t.device, generator=torch.Generator(device=t.device).manual_seed(2))
    g[:, bad] = 0.0
    keep = torch.ones(wl.npt, dtype=torch.bool, device=t.device)
    keep[bad] = False
    for npv in (2, 40):   # groups of 32 and of 128 times
        q, gq = p[:npv].contiguous(), g[:npv].contiguous()
        f, ref = m.evaluate(t2, q), m.evaluate(t, q)
        assert bool((ref[:, keep] < 1).any()) and torch.equal(f[:, keep], ref[:, keep])
        ga, gb = m.evaluate_grad(t2, q, gq), m.evaluate_grad(t, q, gq)
        assert bool(((ga - gb).abs() <= 1e-12 * gb.abs().amax(0)).all())
        ws = m.prepare(t2, q)
        fb, _ = m.evaluate_both(t2, q, gq, ws)
        assert torch.equal(fb, f)
    m.sync_status()
