"""Workspaces and scratch of larger batches serve smaller ones, with the same bits.

A small batch's gradient takes more partial sums (a launch cut below the chunks) than its share of a large one;
given only the large batch's bytes, or a ragged last chunk of the staged host path, it runs uncut.
"""
import ctypes

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


@pytest.mark.parametrize("precision,npb,ss", [("mixed", 1, (1,)), ("mixed", 2, (1, 5)), ("fp64", 1, (1,)), ("fp64", 1, (3,))])
def test_workspace_of_a_larger_batch(rr, precision, npb, ss):
    import torch
    wl = W.make_small("quadratic", npv=1500, npt=12000, npb=npb, ss=ss, exptime=(0.02,) * npb, seed=3, precision=precision, span=9.0)
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    g = torch.randn((wl.npv, wl.npt), device=t.device, generator=torch.Generator(device=t.device).manual_seed(4)).to(m.dtype)
    larger = 0
    sizes = {k: m.workspace_bytes(k, wl.npt, True) for k in range(1, wl.npv)}
    # the batch that falls shortest of a larger one's workspace: the last before the uncut launches
    worst = max(range(1, 1499), key=lambda k: sizes[k] - sizes[k + 1])
    for npv in (1, 40, 300, worst, 1400):
        need, big = m.workspace_bytes(npv, wl.npt, True), m.workspace_bytes(npv + 1, wl.npt, True)
        q, gq = p[:npv].contiguous(), g[:npv].contiguous()
        ref = m.evaluate_grad(t, q, gq, pb, wl.supersampling, wl.exptime)
        f = m.evaluate(t, q, pb, wl.supersampling, wl.exptime)
        for n in sorted({min(m.workspace_bytes(k, wl.npt, True) for k in range(npv, 1500)), need, big}):
            larger += n < need
            ws = torch.empty(n, dtype=torch.uint8, device=t.device)
            out = m.evaluate_grad(t, q, gq, pb, wl.supersampling, wl.exptime, workspace=ws)
            assert torch.equal(out, ref)
            m.prepare(t, q, pb, wl.supersampling, wl.exptime, workspace=ws)
            fb, gb = m.evaluate_both(t, q, gq, ws, pb, wl.supersampling, wl.exptime)
            assert torch.equal(gb, ref) and torch.equal(fb, f)
    m.sync_status()
    assert precision == "fp64" or larger > 0   # the case was met


def test_staged_host_path_with_a_small_last_chunk(rr):
    import torch
    wl = W.make_small("quadratic", npv=831, npt=20000, seed=3, span=9.0)
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    g = np.random.default_rng(2).standard_normal((wl.npv, wl.npt)).astype(np.float32)
    ref = m.evaluate_grad(t, p, torch.as_tensor(g, device=t.device))
    f, go = np.empty((wl.npv, wl.npt), np.float32), np.empty((wl.npv, m.nparam))
    ss, ex = np.ones(1, np.int32), np.zeros(1)

    def ptr(a):
        return ctypes.c_void_p(a.ctypes.data)
    times, params = np.ascontiguousarray(wl.times), np.ascontiguousarray(wl.params)
    for chunk in (800, 500):
        st = m.lib.rr_evaluate_host(m._h, ptr(times), None, wl.npt, ptr(params), wl.npv, ss.ctypes.data, ex.ctypes.data, ptr(g),
                                    ptr(f), ptr(go), None, chunk)
        m._check(st)
        assert np.array_equal(go, ref.cpu().numpy())
