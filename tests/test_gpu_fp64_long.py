"""FP64 series of more than 67 million times: light curves and gradient beyond 65,535 chunks of 1,024 times.

The stretches compared are the same bits as evaluations of those times alone; a cotangent that is zero outside a
stretch gives the gradient of that stretch (another order of the FP64 sums: 1e-12 of the largest component).
"""
import numpy as np
import pytest

from paper_2009_08500_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_more_than_65535_chunks():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2009_08500_gb300 import rr
    n = 65535 * 1024 + 90_001
    wl = W.make_small("quadratic", npv=1, npt=8, precision="fp64", seed=5)
    m = rr.model_for(wl)
    p = torch.as_tensor(wl.params, device="cuda")
    t = torch.arange(n, dtype=torch.float64, device="cuda") * 1e-4
    f = m.evaluate(t, p)
    for a, b in ((0, 60_000), (40_000_000, 40_050_000), (n - 90_001, n)):
        part = m.evaluate(t[a:b].contiguous(), p)
        assert torch.equal(part, f[:, a:b]) and bool((part < 1).any())
    a, b = n - 50_000, n
    g = torch.zeros((1, n), dtype=torch.float64, device="cuda")
    g[:, a:b] = torch.as_tensor(np.random.default_rng(1).normal(size=(1, b - a)), device="cuda")
    ref = m.evaluate_grad(t[a:b].contiguous(), p, g[:, a:b].contiguous())
    out = m.evaluate_grad(t, p, g)
    assert float((out - ref).abs().max()) <= 1e-12 * float(ref.abs().max()) and float(ref.abs().max()) > 0
    ws = m.prepare(t, p)
    fb, gb = m.evaluate_both(t, p, g, ws)
    assert torch.equal(fb, f) and torch.equal(gb, out)
    m.sync_status()
