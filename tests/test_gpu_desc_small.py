"""The f64 descriptor calls where the kernels change over -- small shapes and few columns stay on the FP64 pipe, a warp per
atom -- and that small shapes cost no more than that (GPU)."""
import numpy as np
import pytest
import torch

import workloads as W
from gpu_common import lib, need_gpu, product_model, to_dev

pytestmark = pytest.mark.gpu
LD = np.longdouble
EPS = LD(2) ** -53


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


# both sides of the rules' lines, and the ends of their ranges
@pytest.mark.parametrize("M1,M2", [(1, 1), (35, 4), (36, 4), (48, 3), (512, 4), (513, 10), (550, 11), (600, 12), (1816, 1)])
def test_descriptor_on_both_sides(M1, M2):
    rng = np.random.default_rng(M1)
    T = rng.normal(size=(21, 4, M1)) * 2.0 ** -rng.integers(0, 30, size=(21, 1, M1))
    D = lib().dp_descriptor_contract(torch.from_numpy(T).cuda(), M2).cpu().numpy()
    t = T.astype(LD)
    ref = np.einsum("ikm,ikn->imn", t, t[:, :, :M2])
    mag = np.einsum("ikm,ikn->imn", np.abs(t), np.abs(t[:, :, :M2]))
    assert (np.abs(D - ref) <= 4 * EPS * mag).all()


@pytest.mark.parametrize("M1,M2", [(1, 1), (20, 3), (32, 15), (32, 16), (79, 6), (80, 6), (22, 22), (23, 23)])
def test_backward_on_both_sides(M1, M2):
    rng = np.random.default_rng(M1)
    T, dD = rng.normal(size=(21, 4, M1)), rng.normal(size=(21, M1, M2))
    dT = lib().dp_descriptor_contract_grad(torch.from_numpy(T).cuda(), torch.from_numpy(dD).cuda()).cpu().numpy()
    t, d = T.astype(LD), dD.astype(LD)
    ref = np.einsum("imn,ikn->ikm", d, t[:, :, :M2])
    ref[:, :, :M2] += np.einsum("imn,ikm->ikn", d, t)
    bound = (M1 + M2) * EPS * np.abs(d).max(axis=(1, 2))[:, None, None] * np.abs(t).max(axis=2)[:, :, None]
    assert (np.abs(dT - ref) <= bound).all()


@pytest.mark.parametrize("M1,M2", [(32, 4), (36, 4), (20, 3)])
def test_the_forward_writes_the_calls_bits(M1, M2):
    dpc = lib()
    w = W.water(seed=57, nmol=40, widths=(1, M1 // 4, M1 // 2, M1), M2=M2, sel=(39, 77), rc=5.2)
    m, x = product_model(w, torch.float64), to_dev(w, torch.float64)
    plan = dpc.dp_tabulate_tc_plan_f64(m.table, m.info, w.nnei)
    T, D = dpc.dp_tabulate_fusion_fwd_tc_f64(plan, m.info, x["s"], x["Rt"], x["nvalid"], x["atype"], w.sel, M2=M2)
    assert torch.equal(D.view(torch.int64), dpc.dp_descriptor_contract(T, M2).view(torch.int64))


def _us(call):
    best = np.inf
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(10):
            call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 100)
    return best


@pytest.mark.parametrize("M1,M2", [(1, 1), (8, 2), (16, 4)])
def test_small_shapes_cost_a_warp_an_atom(M1, M2):
    """200,000 atoms in f64 against the f32 calls, a warp per atom as well: twice the memory and a few FP64 operations (D 1.3,
    1.3 and 1.9 times the f32 calls, dT 1.4, 2.1 and 2.5); a block per atom took 3.1 to 3.2 times, and dT 6.1 to 8.6."""
    dpc = lib()
    T, dD = torch.randn(200000, 4, M1, device="cuda"), torch.randn(200000, M1, M2, device="cuda")
    T64, dD64 = T.double(), dD.double()
    o = [torch.empty_like(a) for a in (dD, T, dD64, T64)]
    d32, d64 = (_us(lambda a=a, b=b: dpc.dp_descriptor_contract(a, M2, out=b)) for a, b in ((T, o[0]), (T64, o[2])))
    t32, t64 = (_us(lambda a=a, g=g, b=b: dpc.dp_descriptor_contract_grad(a, g, out=b))
                for a, g, b in ((T, dD, o[1]), (T64, dD64, o[3])))
    assert d64 <= 2.4 * d32 and t64 <= 3.6 * t32, (d32, d64, t32, t64)
