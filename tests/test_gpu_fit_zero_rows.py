"""Rows of zeros in the fitting net's GEMMs -- atoms without a gradient, padding -- cost nothing (GPU): timed beside the
same call without them, since the values cannot tell.  What must leave the common path still does: a column or a row
with a NaN beside zeros, and products below the normal range."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_common import lib, need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _us(*calls):
    """The least of several timings of each call, taken in turn."""
    best = [np.inf] * len(calls)
    for _ in range(8):
        for i, call in enumerate(calls):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                call()
            b.record()
            torch.cuda.synchronize()
            best[i] = min(best[i], a.elapsed_time(b) * 200)
    return best


def test_atoms_without_a_gradient_cost_nothing():
    dpc = lib()
    widths, n = [512, 240, 240, 240, 1], 12288
    params = torch.from_numpy(W.net_params(3, widths, 1)).cuda()
    D = torch.from_numpy(W.normal(8, (n, widths[0]), 0.0, 0.3)).cuda()
    ts = np.array([0, n], np.int64)
    work = torch.empty(dpc.dp_fitting_tc_work_bytes(widths, n), dtype=torch.uint8, device="cuda")
    E, act = dpc.dp_fitting_fwd_tc_f64(params, widths, ts, D, work=work)
    g = torch.ones(n, dtype=torch.float64, device="cuda")
    masked = g.clone()
    masked[::32] = 0.0
    t = _us(*(lambda x=x: dpc.dp_fitting_grad_tc_f64(params, widths, ts, act, g=x, work=work) for x in (g, masked)))
    assert t[1] <= 1.1 * t[0], t  # (1.21 before)
    a = dpc.dp_fitting_grad_tc_f64(params, widths, ts, act, g=masked, work=work)
    assert not a[::32].any() and a[1::32].any()


def test_nans_beside_zeros_and_small_products():
    dpc = lib()
    widths, n = [32, 64, 64, 1], 160  # the last tile a quarter full
    params = torch.from_numpy(W.net_params(3, widths, 1)).cuda()
    ts = np.array([0, n], np.int64)
    D = torch.from_numpy(W.normal(8, (n, 32), 0.0, 0.3)).cuda()
    D[3], D[140] = 0.0, 0.0
    D[7, 5] = float("nan")
    p = params.clone().reshape(-1)
    p[10] = float("inf")  # W_1[0][10]: column 10 of the first layer
    E, act = dpc.dp_fitting_fwd_tc_f64(p.reshape(params.shape), widths, ts, D)
    torch.cuda.synchronize()
    a = act[:, :64]
    assert torch.isnan(a[7]).all() and torch.isnan(a[:, 10]).all()
    keep = [i for i in range(n) if i != 7]
    cols = [c for c in range(64) if c != 10]
    assert torch.isfinite(a[keep][:, cols]).all()
    # z = D W + b below the normal range: tanh z = z to the bit, and z an exact sum rounded once
    small = torch.zeros_like(D)
    small[:, 0] = 2.0 ** -1000
    q = torch.zeros_like(p)
    q[:64] = torch.arange(1, 65, dtype=torch.float64).cuda() * 2.0 ** -70  # W_1[0][n]
    q[65] = 2.0 ** -3  # W_1[1][1]
    small[9, 0], small[9, 1] = 0.0, 2.0 ** -900
    E, act = dpc.dp_fitting_fwd_tc_f64(q.reshape(params.shape), widths, ts, small)
    torch.cuda.synchronize()
    ref = small.cpu().numpy()[:, :2].astype(np.longdouble) @ np.stack([q[:64].cpu().numpy(), q[64:128].cpu().numpy()])
    got, ref = act[:, :64].cpu().numpy(), ref.astype(np.float64)
    ref[:, 1] = np.where(np.arange(n) == 9, ref[:, 1], 0.0)  # (2^-69 beside 2^-3 in one column of W: below its 55 places)
    assert np.array_equal(got, ref)
