"""dp_env_mat_f64's rows at the edges of its arithmetic (1/r from the float root by one step, the switch in fixed
point) against extended precision on the host: r just below and above rcs and rc, scales where the float root
serves and where it does not, both switches, normalised and not (GPU).  Bound: 1/r and s within 4 units of the last
place of their largest factor; in the switch's tail the value itself is small and its error that of w near 1."""
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
@pytest.mark.parametrize("norm", [None, (0.125, 0.5, 2.0)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 40, 2.0 ** -45, 2.0 ** 60, 2.0 ** -60])
def test_rows_at_the_edges(kind, norm, scale):
    dpc = lib()
    rcs, rc = 2.0 * scale, 8.0 * scale
    rng = np.random.default_rng(5)
    edges = [np.nextafter(x * scale, s) for x in (2.0, 8.0) for s in (0.0, np.inf)]
    r = np.concatenate([[0.3 * scale, 1.9999 * scale, rcs, rc, 7.9999999 * scale, 5.0 * scale], edges,
                        rng.uniform(0.2, 8.5, 300) * scale])
    d = rng.normal(size=(r.size, 3))
    d = d / np.linalg.norm(d, axis=1, keepdims=True) * r[:, None]
    d[6:10] = np.stack([r[6:10], 0 * r[6:10], 0 * r[6:10]], axis=1)  # exactly these radii
    coord = np.concatenate([np.zeros((1, 3)), d])
    n = r.size
    nlist = np.arange(1, n + 1, dtype=np.int32)[None]
    env = dpc.env_info(rcs, rc, kind, norm)
    s, Rt, nv = dpc.dp_env_mat(torch.from_numpy(coord).cuda(), torch.from_numpy(nlist).cuda(), [n], env)
    torch.cuda.synchronize()
    assert int(nv[0, 0]) == n
    x = d.astype(LD)
    rr = np.sqrt((x * x).sum(1))
    u = (rr - LD(rcs)) / (LD(rc) - LD(rcs))
    pi = LD(4) * np.arctan(LD(1))
    w = u ** 3 * (-6 * u * u + 15 * u - 10) + 1 if kind == 1 else np.cos(pi * u) / 2 + LD(0.5)
    w = np.where(rr < rcs, LD(1), np.where(rr < rc, w, LD(0)))
    mean, std, std_all = (LD(v) for v in (norm or (0.0, 1.0, 1.0)))
    sv = w / rr
    ref = np.concatenate([((sv - mean) / std)[:, None], (sv / rr / std_all)[:, None] * x], axis=1)
    bound = 4 * LD(2) ** -52 * np.concatenate([((1 / rr + abs(mean)) / std)[:, None], (1 / rr / rr / std_all)[:, None]
                                              * abs(x)], axis=1)
    got = Rt[0].cpu().numpy()
    assert np.array_equal(got[:, 0], s[0].cpu().numpy())
    assert (np.abs(got - ref) <= bound).all(), float((np.abs(got - ref) / bound).max())
