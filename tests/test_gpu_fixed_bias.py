"""The fixed-point sums of the f64 path are not biased (GPU): sums over many atoms (the virial, above all) add up
what every row's rounding has in common, so a floor instead of a rounding shows there although each row is exact to
an f64 unit.  The signed errors against extended precision, summed over independent groups, stay within 6 of their
standard deviations (below 1e-8 by chance for unbiased errors)."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_common import lib, need_gpu, product_model, to_dev

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _z(groups):
    g = np.asarray(groups, dtype=np.float64)
    return abs(g.sum()) / np.sqrt((g * g).sum())


def test_descriptor():
    rng = np.random.default_rng(1)
    T = rng.normal(size=(400, 4, 40))
    D = lib().dp_descriptor_contract(torch.from_numpy(T).cuda(), 8)
    torch.cuda.synchronize()
    t = T.astype(LD)
    err = D.cpu().numpy() - np.einsum("ikm,ikn->imn", t, t[:, :, :8])
    assert _z(err[:, 8:].reshape(-1)) <= 6.0  # (m != n)


@pytest.mark.parametrize("M1", [20, 160])  # seven 8-bit digits, nine 6-bit digits
def test_rows(M1):
    w = W.water(seed=57, nmol=60, widths=(1, M1 // 4, M1 // 2, M1), M2=3, sel=(39, 77), rc=5.2)
    m, x = product_model(w, torch.float64), to_dev(w, torch.float64)
    ds, dRt = lib().dp_tabulate_fusion_grad_tc_f64(m.table, m.info, x["s"], x["Rt"], x["nvalid"], x["atype"], w.sel,
                                                   x["dT"])
    torch.cuda.synchronize()
    ds, dRt = ds.cpu().numpy(), dRt.cpu().numpy()
    info, nt, nnei = m.info, len(w.sel), sum(w.sel)
    n0 = round((info.upper - info.lower) / info.stride0)
    nint = n0 + round((info.upper_ext - info.upper) / info.stride1)
    tab = m.table.cpu().numpy().reshape(nt * nt, nint, 3, M1, 2).transpose(0, 1, 3, 2, 4).reshape(nt * nt, nint, M1, 6)
    value, slope = [], []
    for i in range(w.nloc):
        off = 0
        for b in range(nt):
            rows = np.arange(off, off + w.nvalid[i, b])
            off += w.sel[b]
            s = w.s[i, rows]
            rows, s = rows[(s >= info.lower) & (s < info.upper_ext)], s[(s >= info.lower) & (s < info.upper_ext)]
            l = np.where(s < info.upper, np.minimum(((s - info.lower) / info.stride0).astype(int), n0 - 1),
                         n0 + ((s - info.upper) / info.stride1).astype(int))
            node = np.where(l < n0, LD(info.lower) + l * LD(info.stride0), LD(info.upper) + (l - n0) * LD(info.stride1))
            t = (s - node.astype(np.float64)).astype(LD)[:, None]
            c = tab[w.atype[i] * nt + b, l].astype(LD)
            g, dg = c[..., 0], np.zeros_like(c[..., 0])
            for q in range(1, 6):
                dg, g = dg * t + g, g * t + c[..., q]
            dT = w.dT[i].astype(LD).T / nnei
            e = dRt[i, rows] - g @ dT
            f = ds[i, rows] - (w.Rt[i, rows].astype(LD) * (dg @ dT)).sum(1)
            for key in np.unique(l):  # the rows of an interval share its coefficients' roundings
                value += list(e[l == key].sum(0))
                slope.append(f[l == key].sum())
    assert _z(value) <= 6.0 and _z(slope) <= 6.0, (_z(value), _z(slope))
