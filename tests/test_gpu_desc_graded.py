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
