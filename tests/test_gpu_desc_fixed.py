"""The f64 descriptor and its backward in fixed point (csrc/desc_fixed.cuh) at the edges of their shapes and
scales, against extended precision on the host (GPU).  The bound: an operand is off by at most a unit of its
last of 57 (59) places of the largest element, a sum of n products by 3 n such units, and each of its pieces
is rounded once more: below n 2^-53 max|a| max|b|."""
import numpy as np
import pytest
import torch

from gpu_common import lib, need_gpu

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _ref(T, dD):
    M2 = dD.shape[2]
    t, g = T.astype(LD), dD.astype(LD)
    D = np.einsum("ikm,ikn->imn", t, t[:, :, :M2])
    dT = np.einsum("imn,ikn->ikm", g, t[:, :, :M2])
    dT[:, :, :M2] += np.einsum("imn,ikm->ikn", g, t)
    return D, dT


def _run(T, dD):
    d = [torch.from_numpy(x).cuda() for x in (T, dD)]
    D = lib().dp_descriptor_contract(d[0], dD.shape[2])
    dT = lib().dp_descriptor_contract_grad(d[0], d[1])
    torch.cuda.synchronize()
    return D.cpu().numpy(), dT.cpu().numpy()


# one row, ragged pieces of 16, whole pieces, M2 = M1, more columns than threads, the widest staged and wider
@pytest.mark.parametrize("M1,M2", [(1, 1), (15, 4), (16, 16), (17, 17), (60, 7), (100, 16), (128, 33), (150, 140),
                                   (200, 30), (256, 256)])
@pytest.mark.parametrize("scale", [(0, 0), (-300, 250), (500, -500)])
def test_shapes_and_scales(M1, M2, scale):
    rng = np.random.default_rng(M1 * 1000 + M2)
    n = 9
    T = rng.normal(size=(n, 4, M1)) * rng.choice([1.0, 1e-3, 30.0], size=(n, 4, 1)) * 2.0 ** scale[0]
    dD = rng.normal(size=(n, M1, M2)) * 2.0 ** scale[1]
    T[1] = 0.0
    dD[2] = 0.0
    T[3, 2], dD[4, :, M2 // 2] = 0.0, 0.0
    D, dT = _run(T, dD)
    rD, rT = _ref(T, dD)
    mt = np.abs(T).max(axis=2)  # [n][4]
    bD = (4 * 2.0 ** -53) * LD(1) * (mt.max(axis=1).astype(LD) ** 2)[:, None, None] + np.abs(rD) * 2.0 ** -53
    assert (np.abs(D - rD) <= bD).all()
    bT = (M1 + M2) * 2.0 ** -53 * np.abs(dD).max(axis=(1, 2)).astype(LD)[:, None, None] * mt.astype(LD)[:, :, None]
    assert (np.abs(dT - rT) <= bT + np.abs(rT) * 2.0 ** -53).all()


@pytest.mark.parametrize("M1,M2", [(17, 5), (100, 16)])
def test_nonfinite_stays_in_its_elements(M1, M2):
    rng = np.random.default_rng(5)
    T, dD = rng.normal(size=(6, 4, M1)), rng.normal(size=(6, M1, M2))
    clean = _run(T, dD)
    T2, d2 = T.copy(), dD.copy()
    T2[1, 2, M1 - 1], T2[2, 0, 0], T2[3, 1, 1] = np.nan, np.inf, 1e-310
    d2[4, 3, 1] = -np.inf
    with np.errstate(invalid="ignore"):
        rD, rT = _ref(T2, d2)
    D, dT = _run(T2, d2)
    assert np.array_equal(np.isnan(D), np.isnan(rD.astype(float))) and np.array_equal(np.isinf(D), np.isinf(rD))
    assert np.array_equal(np.isfinite(dT), np.isfinite(rT))
    for i in (0, 5):
        assert np.array_equal(D[i], clean[0][i]) and np.array_equal(dT[i], clean[1][i])
    m = np.isfinite(rT[3])
    assert np.abs(dT[3] - rT[3])[m].max() <= (M1 + M2) * 2.0 ** -53 * np.abs(dD[3]).max() * np.abs(T[3]).max()


@pytest.mark.parametrize("M1,M2", [(1, 1), (17, 17), (100, 16), (140, 32), (200, 30)])
def test_df64_calls_give_the_f64_results(M1, M2):
    """The df64 calls' arrays are f64; they run the same kernels wherever those take the shape,
    and refuse what they refused (a backward with M1 (9 + M2) > 7264)."""
    rng = np.random.default_rng(M1)
    T = torch.from_numpy(rng.normal(size=(7, 4, M1))).cuda()
    dD = torch.from_numpy(rng.normal(size=(7, M1, M2))).cuda()
    d = lib()
    assert torch.equal(d.dp_descriptor_contract_df64(T, M2), d.dp_descriptor_contract(T, M2))
    if M1 * (9 + M2) > 7264:
        with pytest.raises(d.DPError):
            d.dp_descriptor_contract_grad_df64(T, dD)
    else:
        assert torch.equal(d.dp_descriptor_contract_grad_df64(T, dD), d.dp_descriptor_contract_grad(T, dD))
