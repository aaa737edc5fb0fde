"""The f64 descriptor calls take as many atoms as four to a block of a grid hold, though their kernels take a block each
(CPU): up to there a call reaches its launch, which fails without a device; from there on it is refused."""
import ctypes

import pytest
import torch

LIMIT = 4 * (2 ** 31 - 1)


@pytest.mark.skipif(torch.cuda.is_available(), reason="the pointers are not memory: only where nothing can be launched")
@pytest.mark.parametrize("arith", ["f64", "df64"])
def test_atoms_above_a_grid(arith):
    import paper_2107_02103_gb300 as dpc
    p = ctypes.c_void_p(4096)
    fwd, grad = getattr(dpc._lib, f"dp_descriptor_contract_{arith}"), getattr(dpc._lib, f"dp_descriptor_contract_grad_{arith}")
    for n in (1, 2 ** 31 - 1, 2 ** 31, LIMIT):
        assert fwd(p, n, 1, 1, p, None) == dpc.DP_ERR_CUDA, n
        assert grad(p, p, n, 1, 1, p, None) == dpc.DP_ERR_CUDA, n
    for n in (LIMIT + 1, 2 ** 40):
        assert fwd(p, n, 1, 1, p, None) == dpc.DP_ERR_SHAPE
        assert grad(p, p, n, 1, 1, p, None) == dpc.DP_ERR_SHAPE
