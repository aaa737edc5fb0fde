"""The fitting net's persistent tensor-core GEMM at the edges of its tiles, shares, types and work buffers (GPU):
against the FP64-pipe net (1e-13, as in test_gpu_fitting_tc), and bit for bit however the work buffer makes it
cut types into batches and rows into chunks -- every output is summed exactly and rounded once."""
import ctypes

import numpy as np
import pytest
import torch

import workloads as W
from gpu_common import lib, need_gpu, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _net(hidden, K, nat, nout=1, seed=3):
    ntypes = len(nat)
    widths = [K, *hidden, nout]
    params = torch.from_numpy(W.net_params(seed, widths, ntypes)).cuda()
    ts = np.concatenate([[0], np.cumsum(nat)]).astype(np.int64)
    n = int(ts[-1])
    D = torch.from_numpy(W.normal(8, (n, K), 0.0, 0.3)).cuda()
    g = torch.from_numpy(W.normal(9, (n,) if nout == 1 else (n, nout))).cuda()
    return params, widths, ts, D, g


# rows around 128, columns around 64, K around a slice, a share (512) and two, shares that split K, eight types
@pytest.mark.parametrize("hidden,K,nat,nout", [
    ((63,), 1, (1,), 1), ((64, 64), 15, (127, 128), 1), ((65, 65, 1), 17, (129, 0, 1), 1), ((33,), 512, (64,), 1),
    ((48,), 513, (130,), 7), ((128, 128), 1030, (3, 5), 64), ((30, 30), 64, (9, 1, 140, 0, 2, 128, 33, 7), 65),
    ((240, 240, 240), 1600, (20, 30), 1)])
def test_tiles_shares_and_types(hidden, K, nat, nout):
    dpc = lib()
    params, widths, ts, D, g = _net(hidden, K, nat, nout)
    E, act = dpc.dp_fitting_fwd_tc_f64(params, widths, ts, D)
    dD = dpc.dp_fitting_grad_tc_f64(params, widths, ts, act, g=g)
    E2, act2 = dpc.dp_fitting_fwd(params, widths, ts, D)
    dD2 = dpc.dp_fitting_grad(params, widths, ts, act2, g=g)
    torch.cuda.synchronize()
    for a, b in ((act, act2), (E, E2), (dD, dD2)):
        assert rel(a.cpu().numpy(), b.cpu().numpy()) <= 1e-13
    assert dpc.dp_tc_wait_timeouts() == 0


@pytest.mark.parametrize("nout", [1, 5])
def test_any_work_buffer_gives_the_same_bits(nout):
    """The queried size, and less by steps down to the smallest accepted: fewer types a batch, fewer rows a chunk."""
    dpc = lib()
    params, widths, ts, D, g = _net((48, 48), 200, (300, 1, 270, 129, 2, 40, 64, 65), nout)
    n = int(ts[-1])
    need = dpc.dp_fitting_tc_work_bytes(widths, n)
    w = (ctypes.c_int32 * len(widths))(*widths)
    start = (ctypes.c_int64 * len(ts))(*[int(x) for x in ts])
    work = torch.empty((need,), dtype=torch.uint8, device="cuda")
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    shape = (n,) if nout == 1 else (n, nout)

    def call(nbytes):
        E, act, dD = (torch.full(s, float("nan"), dtype=torch.float64, device="cuda") for s in (shape, (n, 96), (n, 200)))
        work.fill_(0xff)
        rc = dpc._lib.dp_fitting_fwd_tc_f64(p(params), w, len(widths) - 1, len(ts) - 1, start, p(D), p(E), p(act), p(work),
                                            nbytes, st)
        rc = rc or dpc._lib.dp_fitting_grad_tc_f64(p(params), w, len(widths) - 1, len(ts) - 1, start, p(act), p(g), p(dD),
                                                   p(work), nbytes, st)
        torch.cuda.synchronize()
        return rc, (E, act, dD)

    rc, ref = call(need)
    assert rc == 0
    accepted = 0
    for f in (0.95, 0.9, 0.85, 0.8, 0.7, 0.6, 0.5):
        rc, got = call(int(need * f) // 256 * 256)
        if rc != 0:
            assert rc == dpc.DP_ERR_SHAPE
            continue
        accepted += 1
        for a, b in zip(ref, got):
            assert torch.equal(a.view(torch.int64), b.view(torch.int64)), f
    assert call(4096)[0] == dpc.DP_ERR_SHAPE
