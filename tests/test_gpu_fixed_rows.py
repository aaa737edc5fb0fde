"""The integer arithmetic of the f64 tensor-core path's per-row kernels at the edges of its scales (GPU): it works
on fixed points against powers of two, so a power of two on dE/dT or R~ moves the results' exponents and nothing
else; infs, NaNs and extreme scales leave it for the FP64 pipe and touch no other atom."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_common import lib, need_gpu, product_model, rel, to_dev

pytestmark = pytest.mark.gpu
F64 = torch.float64


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.fixture(scope="module")
def setup():
    need_gpu()
    # 2 types, 39 and 77 rows: batches of 32 with a ragged last one; M1 = 20 and (9 x 6 digits) 160
    out = {}
    for M1 in (20, 160):
        w = W.water(seed=57, nmol=40, widths=(1, M1 // 4, M1 // 2, M1), M2=3, sel=(39, 77), rc=5.2)
        out[M1] = w, product_model(w, F64), to_dev(w, F64)
    return out


def _grad(m, x, w, dT=None, Rt=None):
    return lib().dp_tabulate_fusion_grad_tc_f64(m.table, m.info, x["s"], x["Rt"] if Rt is None else Rt, x["nvalid"],
                                                x["atype"], w.sel, x["dT"] if dT is None else dT)


def _fwd(m, x, w, Rt=None):
    return lib().dp_tabulate_fusion_fwd_tc_f64(m.table, m.info, x["s"], x["Rt"] if Rt is None else Rt, x["nvalid"],
                                               x["atype"], w.sel)


def _same(a, b):
    return torch.equal(a.view(torch.int64), b.view(torch.int64))


@pytest.mark.parametrize("M1", [20, 160])
@pytest.mark.parametrize("s", [-900, -380, -1, 300, 380, 900])  # |s| > 400: the rows leave the integer conversion
def test_powers_of_two(setup, M1, s):
    w, m, x = setup[M1]
    ds, dRt = _grad(m, x, w)
    ds2, dRt2 = _grad(m, x, w, dT=x["dT"] * 2.0 ** s)
    assert _same(ds2, ds * 2.0 ** s) and _same(dRt2, dRt * 2.0 ** s)
    T, T2 = _fwd(m, x, w), _fwd(m, x, w, Rt=x["Rt"] * 2.0 ** s)
    if abs(s) < 700:
        assert _same(T2, T * 2.0 ** s)
    else:  # batches summed on the FP64 pipe: another rounding (a few 2^-53 of the largest)
        assert rel((T2 * 2.0 ** -s).cpu().numpy(), T.cpu().numpy()) <= 1e-14


@pytest.mark.parametrize("M1", [20, 160])
def test_infs_nans_and_zero_columns(setup, M1):
    w, m, x = setup[M1]
    ds, dRt = _grad(m, x, w)
    T = _fwd(m, x, w)
    dT = x["dT"].clone()
    dT[3, 1, M1 // 2] = float("inf")
    dT[5] = 0.0
    dT[7, 2] = 0.0
    g, gR = _grad(m, x, w, dT=dT)
    nv = [int(v) for v in w.nvalid[3]]
    rows = torch.cat([torch.arange(nv[0]), w.sel[0] + torch.arange(nv[1])]).cuda()
    assert torch.isnan(g[3, rows]).all() and torch.isnan(gR[3, rows, 1]).all()
    assert _same(gR[3][:, [0, 2, 3]], dRt[3][:, [0, 2, 3]])
    assert not g[5].any() and not gR[5].any() and not gR[7, :, 2].any()
    keep = [i for i in range(w.nloc) if i not in (3, 5, 7)]
    assert _same(g[keep], ds[keep]) and _same(gR[keep], dRt[keep])
    Rt = x["Rt"].clone()
    Rt[2, 1, 3], Rt[4, 0, 0], Rt[9, 2, 1] = float("nan"), float("-inf"), 1e300
    T2 = _fwd(m, x, w, Rt=Rt)
    assert torch.isnan(T2[2, 3]).all() and torch.isnan(T2[4, 0]).all()
    for i, k in ((2, [0, 1, 2]), (4, [1, 2, 3]), (9, [0, 2, 3])):  # the other columns of those atoms
        assert rel(T2[i, k].cpu().numpy(), T[i, k].cpu().numpy()) <= 1e-14
    keep = [i for i in range(w.nloc) if i not in (2, 4, 9)]
    assert _same(T2[keep], T[keep])
    g, gR = _grad(m, x, w, Rt=Rt)
    assert _same(gR, dRt) and torch.isnan(g[2, 1]) and not torch.isfinite(g[4, 0])
    g[2, 1], g[4, 0], g[9, 2] = ds[2, 1], ds[4, 0], ds[9, 2]
    assert _same(g, ds)


def test_zero_components_stay_zero(setup):
    """A plane of atoms: R~'s z components are zero in every batch, and so are T's z row and its part of ds."""
    w, m, x = setup[20]
    Rt = x["Rt"].clone()
    Rt[..., 3] = 0.0
    T, T0 = _fwd(m, x, w, Rt=Rt), _fwd(m, x, w)
    assert not T[:, 3].any() and _same(T[:, :3], T0[:, :3])


def test_every_nvalid_and_order(setup):
    """Rows in random order (keys met again within a batch of 32 and in later ones) against the sorted rows:
    T within the rounding of its sums, each row's gradients to the bit."""
    w, m, x = setup[20]
    T, (ds, dRt) = _fwd(m, x, w), _grad(m, x, w)
    rng = np.random.default_rng(4)
    perm = np.tile(np.arange(w.nnei), (w.nloc, 1))
    for i in range(w.nloc):
        for off, n in ((0, w.nvalid[i, 0]), (w.sel[0], w.nvalid[i, 1])):
            perm[i, off:off + n] = off + rng.permutation(n)
    p = torch.from_numpy(perm).cuda()
    y = {**x, "s": x["s"].gather(1, p).contiguous(),
         "Rt": x["Rt"].gather(1, p[..., None].expand(-1, -1, 4)).contiguous()}
    assert rel(_fwd(m, y, w).cpu().numpy(), T.cpu().numpy()) <= 1e-14
    g, gR = _grad(m, y, w)
    assert _same(g, ds.gather(1, p)) and _same(gR, dRt.gather(1, p[..., None].expand(-1, -1, 4)))
