"""The fitting net's work buffer from the queried size down to the least that is taken: types in batches, row tiles in
chunks, the same bits (GPU) -- every output is summed exactly and rounded once.  The shapes are ones whose least size lies
below the query: with a small system the query counts eight types' planes; with a wide layer and many atoms the least
size holds half of the row tiles."""
import ctypes

import numpy as np
import pytest
import torch

import workloads as W
from gpu_common import lib, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,nat,nout", [
    ((240, 240, 240), (20, 1, 40, 31, 0, 30, 33, 37), 1), ((240, 240, 240), (20, 1, 40, 31, 0, 30, 33, 37), 5),
    ((1024,), (900, 0, 1100), 1), ((1024,), (2000,), 5)])
def test_down_to_the_least_buffer(hidden, nat, nout):
    need_gpu()
    dpc = lib()
    K, ntypes = 1600, len(nat)
    widths = [K, *hidden, nout]
    params = torch.from_numpy(W.net_params(3, widths, ntypes)).cuda()
    ts = np.concatenate([[0], np.cumsum(nat)]).astype(np.int64)
    n, H = int(ts[-1]), sum(hidden)
    D = torch.from_numpy(W.normal(8, (n, K), 0.0, 0.3)).cuda()
    g = torch.from_numpy(W.normal(9, (n,) if nout == 1 else (n, nout))).cuda()
    need = dpc.dp_fitting_tc_work_bytes(widths, n)
    w = (ctypes.c_int32 * len(widths))(*widths)
    start = (ctypes.c_int64 * len(ts))(*[int(x) for x in ts])
    work = torch.empty((need,), dtype=torch.uint8, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)

    def call(nbytes):
        E, act, dD = (torch.full(s, float("nan"), dtype=torch.float64, device="cuda")
                      for s in ((n,) if nout == 1 else (n, nout), (n, H), (n, K)))
        work.fill_(0xff)
        rc = dpc._lib.dp_fitting_fwd_tc_f64(p(params), w, len(widths) - 1, ntypes, start, p(D), p(E), p(act), p(work),
                                            nbytes, st)
        rc = rc or dpc._lib.dp_fitting_grad_tc_f64(p(params), w, len(widths) - 1, ntypes, start, p(act), p(g), p(dD),
                                                   p(work), nbytes, st)
        torch.cuda.synchronize()
        return rc, (E, act, dD)

    rc, ref = call(need)
    assert rc == 0 and all(torch.isfinite(a).all() for a in ref)
    lo, hi = 0, need  # refused, taken
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        rc, got = call(mid)
        assert rc in (0, dpc.DP_ERR_SHAPE)
        lo, hi = (lo, mid) if rc == 0 else (mid, hi)
    assert hi < 0.7 * need
    accepted = 0
    for nbytes in (hi, hi + (need - hi) // 5, hi + (need - hi) // 2, need - 1):
        rc, got = call(nbytes)
        assert rc == 0
        accepted += 1
        for a, b in zip(ref, got):
            assert torch.equal(a.view(torch.int64), b.view(torch.int64)), nbytes
    assert accepted == 4 and call(lo)[0] == dpc.DP_ERR_SHAPE
    assert dpc.dp_tc_wait_timeouts() == 0
