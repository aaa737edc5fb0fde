"""A NaN coordinate, whatever its sign and payload, makes a row with s = 0 and no finite component of R~ but that, as a
comparison with the cut-off that fails does, and touches no other row (GPU)."""
import numpy as np
import pytest
import torch

from gpu_common import lib, need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("bits", [0x7ff8000000000000, 0xfff8000000000000, 0x7ff8000000000123, 0xfff8000000000123])
def test_nan_coordinate(kind, bits):
    need_gpu()
    dpc = lib()
    c = np.zeros((4, 3))
    c[1, 0], c[2, 0], c[3, 1] = 1.0, 3.0, 2.0
    nl = torch.tensor([[1, 2, 3]], dtype=torch.int32).cuda()
    env = dpc.env_info(0.5, 6.0, kind)
    s0, R0, _ = dpc.dp_env_mat(torch.from_numpy(c).cuda(), nl, [3], env)
    c.view(np.uint64)[2, 1] = bits
    s, R, _ = dpc.dp_env_mat(torch.from_numpy(c).cuda(), nl, [3], env)
    torch.cuda.synchronize()
    assert s[0, 1] == 0.0 and R[0, 1, 0] == 0.0 and torch.isnan(R[0, 1, 1:]).all()
    assert torch.equal(s[0, ::2], s0[0, ::2]) and torch.equal(R[0, ::2], R0[0, ::2])
