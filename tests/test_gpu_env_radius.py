"""The radius that the environment kernels form, to the last bit, seen through a switch so narrow that a unit of the
last place of r moves it (GPU).  On an axis r = sqrt(x^2) is x for any square root rounded within half a unit.  Then
u = (x - rcs)/(rc - rcs) is off by 1.5 2^-52 (the subtraction is exact), the switch by 2^-55 of what u gives, and s = w/r
by two roundings: below |w'| 3 2^-53 + 2^-54 + 2 2^-53 w, over r."""
import numpy as np
import pytest
import torch

from gpu_common import lib, need_gpu

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("rc", [0.7, 1.0, 6.0, 8.0, 1e9])
def test_radius_to_the_bit(kind, rc):
    dpc = lib()
    n, rcs = 20000, rc * (1 - 2.0 ** -22)
    x = np.random.default_rng(3).uniform(rcs, rc, n)
    coord = np.zeros((n + 1, 3))
    coord[1:, 1] = x
    nl = torch.arange(1, n + 1, dtype=torch.int32).cuda()[None]
    s, _, _ = dpc.dp_env_mat(torch.from_numpy(coord).cuda(), nl, [n], dpc.env_info(rcs, rc, kind))
    torch.cuda.synchronize()
    r, iw, pi = x.astype(LD), 1 / (LD(rc) - LD(rcs)), LD(4) * np.arctan(LD(1))
    u = (r - LD(rcs)) * iw
    if kind == 1:
        w, dw = u ** 3 * (-6 * u * u + 15 * u - 10) + 1, -30 * u * u * (u - 1) ** 2
    else:
        w, dw = np.cos(pi * u) / 2 + LD(0.5), -pi / 2 * np.sin(pi * u)
    eps = LD(2) ** -53
    bound = (3 * eps * abs(dw) + eps / 2 + 2 * eps * w) / r
    err = np.abs(s[0].cpu().numpy() - w / r)
    assert (err <= bound).all(), float((err / bound).max())
