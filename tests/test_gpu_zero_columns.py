"""Atoms whose dE/dT has a component of zeros (a plane of atoms, a masked gradient) take the rows kernel's fast
conversion like any other (GPU): timed beside the same atoms without the zeros, since the values cannot tell."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_common import lib, need_gpu, product_model, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _rows_us(dpc, call):
    """The rows kernel of one backward: the events around it, the least of several calls."""
    best = np.inf
    for it in range(12):
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(32)]
        dpc.dp_profile_begin(ev)
        call()
        names = dpc.dp_profile_end()
        torch.cuda.synchronize()
        at = names.index("tc_rows")
        if it > 2:
            best = min(best, ev[at - 1].elapsed_time(ev[at]) * 1e3)
    return best


@pytest.mark.parametrize("M1", [100, 160])  # seven 8-bit digits, nine 6-bit digits
def test_zero_columns_cost_nothing(M1):
    dpc = lib()
    w = W.water(seed=57, nmol=700, widths=(1, M1 // 4, M1 // 2, M1), M2=3, sel=(46, 92), rc=6.0)
    m, x = product_model(w, torch.float64), to_dev(w, torch.float64)
    plan = dpc.dp_tabulate_tc_plan_f64(m.table, m.info, w.nnei)

    def backward(dT):
        return lambda: dpc.dp_tabulate_fusion_grad_tc_f64(plan, m.info, x["s"], x["Rt"], x["nvalid"], x["atype"], w.sel, dT)

    plain = _rows_us(dpc, backward(x["dT"]))
    one, some, least = x["dT"].clone(), x["dT"].clone(), x["dT"].clone()
    one[:, 3], some[::8] = 0.0, 0.0
    for dT in (one, some):
        assert _rows_us(dpc, backward(dT)) <= 1.15 * plain
    # what is not zero stays: a column of subnormals against the same scaled up by a power of two
    least[:, 3] = 0.0
    least[5, 3] = torch.from_numpy(np.random.default_rng(1).integers(1, 1 << 20, M1) * 5e-324).cuda()
    up = least.clone()
    up[5, 3] *= 2.0 ** 600
    a, b = backward(least)(), backward(up)()
    assert torch.allclose(a[1][5, :, 3] * 2.0 ** 600, b[1][5, :, 3], rtol=0, atol=1e-3 * float(b[1][5, :, 3].abs().max()))
    assert b[1][5, :, 3].any() and a[1][5, :, 3].any()
