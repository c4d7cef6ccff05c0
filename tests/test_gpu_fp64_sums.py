"""FP64 light curves with sub-exposures: the same bits in every batch.

The FP64 kernel takes groups of 32 or of 128 times by the size of the launch; a time's sub-exposures are added in an
order of their indices alone, so one vector alone, a sub-batch, the whole batch and the staged host path (chunks, a
small last one) give the same bits.
"""
import ctypes

import numpy as np
import pytest

from paper_2009_08500_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CASES = [dict(npt=3001, ss=(10,), exptime=(0.02,)), dict(npt=2500, npb=3, ss=(1, 4, 9), exptime=(0.0, 0.01, 0.02)),
         dict(npt=2000, ss=(33,), exptime=(0.02,)),
         dict(npt=1500, npb=2, ss=(150, 3), exptime=(0.02, 0.01))]


@pytest.fixture(scope="module")
def rr():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2009_08500_gb300 import rr as _rr
    _rr.load_library()
    return _rr


@pytest.mark.parametrize("case", CASES, ids=lambda c: str(c["ss"]))
def test_light_curves_do_not_depend_on_the_batch(rr, case):
    import torch
    wl = W.make_small("quadratic", npv=700, seed=6, precision="fp64", span=9.0, **case)
    m = rr.model_for(wl)
    t, pb, p = rr.to_device(wl)
    ss, ex = wl.supersampling, wl.exptime
    f = m.evaluate(t, p, pb, ss, ex)
    assert bool((f < 1).any())
    for lo, n in ((0, 1), (17, 1), (100, 9), (300, 90), (200, 400)):
        q = p[lo:lo + n].contiguous()
        assert torch.equal(m.evaluate(t, q, pb, ss, ex), f[lo:lo + n])
        ws = m.prepare(t, q, pb, ss, ex)
        assert torch.equal(m.evaluate(t, q, pb, ss, ex, prepared=ws), f[lo:lo + n])
    m.sync_status()
    # the staged host path: chunks below and above the group width's line, and a last chunk of a few vectors
    times, params = np.ascontiguousarray(wl.times), np.ascontiguousarray(wl.params)
    pbi = np.ascontiguousarray(wl.pb_index, np.int32)
    ssa, exa = np.ascontiguousarray(ss, np.int32), np.ascontiguousarray(ex, np.float64)

    def ptr(a):
        return ctypes.c_void_p(a.ctypes.data)
    for chunk in (40, 693):
        out = np.empty((wl.npv, wl.npt))
        m._check(m.lib.rr_evaluate_host(m._h, ptr(times), ptr(pbi) if wl.npb > 1 else None, wl.npt, ptr(params), wl.npv,
                                        ssa.ctypes.data, exa.ctypes.data, None, ptr(out), None, None, chunk))
        assert np.array_equal(out, f.cpu().numpy())
