"""Workspaces of longer series serve shorter ones (fewer vectors or not), with the same bits.

The FP32 adjoint's chunks grow with the number of times, so that partial sums are fewer right behind each step (15 chunks
at 15,360 times, 8 at 15,361); the sizes cover every shorter series all the same.
"""
import pytest

from paper_2009_08500_gb300 import workloads as W

pytestmark = pytest.mark.gpu

STEPS = [(15_360, 15_361), (15_360, 16_384), (15_000, 20_000), (23_000, 25_000), (4_000, 15_361), (130_000, 131_200)]


@pytest.mark.parametrize("precision,npb,ss", [("mixed", 1, (1,)), ("mixed", 3, (1, 5, 2)), ("fp64", 1, (1,))])
def test_workspace_of_a_longer_series(precision, npb, ss):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2009_08500_gb300 import rr
    wl = W.make_small("quadratic", npv=1200, npt=25_000, npb=npb, ss=ss, exptime=(0.01,) * npb, seed=3, precision=precision, span=20.0)
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    t, pb = torch.cat([t] * 6), torch.cat([pb] * 6)
    g = torch.randn(p.shape[0] * 25_000, device=t.device, generator=torch.Generator(device=t.device).manual_seed(4)).to(m.dtype)
    for short, long in STEPS:
        for npv, most in ((1200, 1200), (1000, 1200), (3, 1200), (150, 160)):
            if npv * short > g.numel():
                continue
            ws = torch.empty(m.workspace_bytes(most, long, True), dtype=torch.uint8, device=t.device)
            ts, pbs, q = t[:short].contiguous(), pb[:short].contiguous(), p[:npv].contiguous()
            gq = g[:npv * short].view(npv, short)
            ref = m.evaluate_grad(ts, q, gq, pbs, wl.supersampling, wl.exptime)
            assert torch.equal(m.evaluate_grad(ts, q, gq, pbs, wl.supersampling, wl.exptime, workspace=ws), ref)
            m.prepare(ts, q, pbs, wl.supersampling, wl.exptime, workspace=ws)
            assert torch.equal(m.evaluate_both(ts, q, gq, ws, pbs, wl.supersampling, wl.exptime)[1], ref)
            need = m.lib.rr_request_bytes(m._h, npv, short, 1)
            assert m.lib.rr_request_bytes(m._h, most, long, 1) >= need or npv < most   # (a cut launch's own may be larger)
    m.sync_status()
