"""Runs reused from a forward on other rows (DP_TC_REUSE_RUNS against its contract): a row whose interval its atom's
runs do not hold gets NaN, not another slot's coefficients; the others are as without the change (GPU)."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_common import lib, need_gpu, product_model, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M1", [20, 160])
def test_a_row_without_a_slot_is_nan(M1):
    need_gpu()
    dpc = lib()
    w = W.water(seed=57, nmol=40, widths=(1, M1 // 4, M1 // 2, M1), M2=3, sel=(39, 77), rc=5.2)
    m, x = product_model(w, torch.float64), to_dev(w, torch.float64)
    plan = dpc.dp_tabulate_tc_plan_f64(m.table, m.info, w.nnei)
    work = torch.empty(dpc.dp_tabulate_tc_work_bytes(m.info, w.nloc, w.nnei, len(w.sel), M1), dtype=torch.uint8,
                       device="cuda")
    a = (plan, m.info, x["s"], x["Rt"], x["nvalid"], x["atype"], w.sel)
    dpc.dp_tabulate_fusion_fwd_tc_f64(*a, work=work)
    ds, dRt = dpc.dp_tabulate_fusion_grad_tc_f64(*a, x["dT"], work=work, flags=dpc.DP_TC_REUSE_RUNS)
    s = x["s"].clone()
    for i, q in ((0, 0), (7, 1)):  # of the first type's rows: into an interval that none of them uses
        used = set(((w.s[i, :w.nvalid[i, 0]] - m.info.lower) / m.info.stride0).astype(int).tolist())
        free = next(l for l in range(100) if l not in used)
        s[i, q] = m.info.lower + (free + 0.5) * m.info.stride0
    dpc.dp_tabulate_fusion_fwd_tc_f64(*a, work=work)
    g, gR = dpc.dp_tabulate_fusion_grad_tc_f64(plan, m.info, s, *a[3:], x["dT"], work=work, flags=dpc.DP_TC_REUSE_RUNS)
    torch.cuda.synchronize()
    for i, q in ((0, 0), (7, 1)):
        assert torch.isnan(g[i, q]) and torch.isnan(gR[i, q]).all()
    g[0, 0], g[7, 1], gR[0, 0], gR[7, 1] = ds[0, 0], ds[7, 1], dRt[0, 0], dRt[7, 1]
    assert np.array_equal(g.cpu().numpy(), ds.cpu().numpy()) and np.array_equal(gR.cpu().numpy(), dRt.cpu().numpy())
