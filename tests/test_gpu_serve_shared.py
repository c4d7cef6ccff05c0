"""Requests served beside others launch whole chunks, lone calls cut ones: the same bits.

Small requests of several passbands and exposure lengths (the whole launches go through the time chunks heaviest first),
with and without gradient, submitted at once to the library's server and compared with evaluations alone.
"""
import numpy as np
import pytest

from paper_2009_08500_gb300 import workloads as W
from paper_2009_08500_gb300.serve import NativeServer, ServeRequest

pytestmark = pytest.mark.gpu


def test_whole_launches_beside_others():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2009_08500_gb300 import rr
    spec = dict(npb=3, ss=(1, 4, 9), exptime=(0.0, 0.01, 0.02))
    m = rr.model_for(W.make_small("quadratic", npv=1, npt=8, **spec))
    rng = np.random.default_rng(8)
    wls = [W.make_small("quadratic", npv=int(rng.integers(1, 40)), npt=int(rng.integers(200, 40_000)), seed=i, span=8.0, **spec)
           for i in range(24)]
    pin = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a, dt)).pin_memory()  # noqa: E731
    reqs = []
    for i, wl in enumerate(wls):
        g = pin(rng.normal(size=(wl.npv, wl.npt)), np.float32) if i % 2 else None
        out = {"flux": torch.empty((wl.npv, wl.npt), dtype=torch.float32).pin_memory(),
               "status": torch.empty(wl.npv, dtype=torch.int32).pin_memory()}
        if g is not None:
            out["grad"] = torch.empty((wl.npv, m.nparam), dtype=torch.float64).pin_memory()
        reqs.append(ServeRequest(fit=0, times=pin(wl.times, np.float64), params=pin(wl.params, np.float64),
                                 pb_index=pin(wl.pb_index, np.int32), supersampling=wl.supersampling, exptime=wl.exptime,
                                 grad_flux=g, out=out))
    with NativeServer({0: m}, slots=8, mem_budget=4 << 30) as srv:
        for f in [srv.submit(r) for r in reqs]:
            f.result(timeout=120)
        assert srv.stats()["max_inflight"] > 1
    for wl, r in zip(wls, reqs):
        t, pb, p = rr.to_device(wl)
        assert np.array_equal(r.out["flux"].numpy(), m.evaluate(t, p, pb, wl.supersampling, wl.exptime).cpu().numpy())
        if r.grad_flux is not None:
            g = m.evaluate_grad(t, p, r.grad_flux.to(t.device), pb, wl.supersampling, wl.exptime)
            assert np.array_equal(r.out["grad"].numpy(), g.cpu().numpy())
