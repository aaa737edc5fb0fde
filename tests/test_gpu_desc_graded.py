"""The f64 descriptor and its backward on channels of very different sizes, element by element against extended
precision on the host (GPU).

D[m][n] is a sum of four products.  Either it is taken in fixed point, and then each of its four terms is off by at
most 1.25 units (half a unit of 60 places from either factor, a quarter for the product of the low limbs) and the
sum by half a unit more, 5.5 in all, on sums of at least 1.84 2^53 units (less than 3 2^-53 of the sum of
magnitudes), and is rounded once; or by one multiplication and three FMAs.  Both stay below
4 2^-53 sum_k |T[k][m] T[k][n]|."""
import numpy as np
import pytest
import torch

from gpu_common import lib, need_gpu

pytestmark = pytest.mark.gpu
LD = np.longdouble
EPS = LD(2) ** -53


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _T(kind, n, M1, rng):
    T = rng.normal(size=(n, 4, M1))
    if kind == "graded":  # channels from 1 down to 2^-40
        T *= 2.0 ** -rng.integers(0, 41, size=(n, 1, M1))
    elif kind == "crossed":  # half of the channels live in k = 0, half in k = 1, and only just in the other
        T[:, 0, ::2] *= 2.0 ** -30
        T[:, 1, 1::2] *= 2.0 ** -30
        T[:, 2:] *= 2.0 ** -45
    elif kind == "isolated":  # zeros of both signs, a channel of zeros, subnormals, and channels out of the range
        T[:, :, ::3] = 0.0
        T[:, 1, 1::3] = -0.0
        T[:, :, M1 // 2] *= 2.0 ** 200
        T[:, :, M1 - 1] = 5e-324
        T[:, 0, 0] = 2.0 ** -1000
    return T


@pytest.mark.parametrize("kind", ["plain", "graded", "crossed", "isolated"])
@pytest.mark.parametrize("M1,M2", [(1, 1), (17, 5), (40, 40), (100, 16), (150, 140)])
def test_descriptor_elementwise(kind, M1, M2):
    rng = np.random.default_rng(M1 + M2)
    T = _T(kind, 33, M1, rng)
    D = lib().dp_descriptor_contract(torch.from_numpy(T).cuda(), M2)
    torch.cuda.synchronize()
    t = T.astype(LD)
    ref = np.einsum("ikm,ikn->imn", t, t[:, :, :M2])
    mag = np.einsum("ikm,ikn->imn", np.abs(t), np.abs(t[:, :, :M2]))
    err = np.abs(D.cpu().numpy() - ref)
    # (results below the normal range are rounded to units of 2^-1074, at most four times)
    assert (err <= 4 * EPS * mag + 4 * LD(2) ** -1074).all(), float((err / np.maximum(mag, LD(2) ** -1000)).max())


def _dD(kind, n, M1, M2, rng):
    dD = rng.normal(size=(n, M1, M2))
    if kind in ("rows", "both"):
        dD *= 2.0 ** -rng.integers(0, 31, size=(n, M1, 1))
    if kind in ("columns", "both"):
        dD *= 2.0 ** -rng.integers(0, 31, size=(n, 1, M2))
    if kind == "zeros":  # between graded rows
        dD *= 2.0 ** -rng.integers(0, 31, size=(n, M1, 1))
        dD[:, ::3], dD[:, :, ::2] = 0.0, -0.0
        dD[1], dD[2, 1:] = 0.0, 0.0
    elif kind == "extreme":  # out of the exponents' range in one way an atom
        for i, e in enumerate((100, -300, -700, -1060)):
            dD[i::5, M1 - 1] *= 2.0 ** e
            dD[i::5, :, 0] *= 2.0 ** (e // 2)
    return dD


@pytest.mark.parametrize("kind", ["plain", "rows", "columns", "both", "zeros", "extreme"])
@pytest.mark.parametrize("Tkind", ["plain", "graded", "isolated"])
@pytest.mark.parametrize("M1,M2", [(1, 1), (17, 5), (40, 40), (100, 16), (70, 64)])
def test_backward_by_rows_and_columns(kind, Tkind, M1, M2):
    """Each row and column of dD against its own largest, R_m C_n >= |dD[m][n]|.  A term of either sum is off by
    1.13 2^-57 of the product of the powers of two above its factors, which are within 8 of R_m C_n |T|: below
    0.6 2^-53 of the largest such product in the sum; the pieces of 16 terms are rounded and added in f64."""
    rng = np.random.default_rng(M1 + M2)
    n = 33
    T, dD = _T(Tkind, n, M1, rng) * rng.choice([1.0, 1e-3, 30.0], size=(n, 4, 1)), _dD(kind, n, M1, M2, rng)
    got = lib().dp_descriptor_contract_grad(torch.from_numpy(T).cuda(), torch.from_numpy(dD).cuda())
    torch.cuda.synchronize()

    def sums(t, d):
        return np.einsum("imn,ikn->ikm", d, t[:, :, :M2]), np.einsum("imn,ikm->ikn", d, t)

    t, d = T.astype(LD), dD.astype(LD)
    a, b = sums(t, d)
    ma, mb = sums(np.abs(t), np.abs(d))
    C = np.abs(d).max(axis=1)
    R = (np.abs(d) / np.where(C > 0, C, 1)[:, None, :]).max(axis=2)
    xa = (C[:, None, :] * np.abs(t[:, :, :M2])).max(axis=2)[:, :, None] * R[:, None, :]  # of dT[k][m]
    xb = (R[:, None, :] * np.abs(t)).max(axis=2)[:, :, None] * C[:, None, :]
    bound = EPS * (M2 * xa + ((M2 + 15) // 16 + 2) * ma)
    a[:, :, :M2] += b
    bound[:, :, :M2] += EPS * (M1 * xb + ((M1 + 15) // 16 + 2) * mb)
    err = np.abs(got.cpu().numpy() - a)
    # (FP64 sums of M1 + M2 terms for what is out of range; units of 2^-1074 below the normal range)
    wild = (M1 + M2) * EPS * ma
    wild[:, :, :M2] += (M1 + M2) * EPS * mb
    bound = np.where(np.isin(np.arange(n) % 5, range(4))[:, None, None], np.maximum(bound, wild), bound) \
        if kind == "extreme" else np.maximum(bound, wild) if Tkind == "isolated" else bound
    assert (err <= bound + (M1 + M2) * LD(2) ** -1074).all()
