"""Left multiplies by more rows than the tensor-core kernels hold (above 384) take the CUDA-core kernel on
every point count, also on multiples of 128."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from paper_2101_03155_gb300 import ace as abi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [384, 385, 420])
@pytest.mark.parametrize("npts", [128, 132, 2560])
def test_many_rows(n, npts):
    import torch

    gen = torch.Generator().manual_seed(n + npts)
    w = torch.randn((n, npts), generator=gen, dtype=torch.float32)
    d = ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n)
    op = abi.ace_build_from_m(d, -torch.eye(n, dtype=torch.float64, device="cuda"), w.cuda())
    xi = torch.from_numpy(abi.get_numpy(op, abi.ACE_GET_XI).reshape(n, npts)).double()
    # the factor is one: products with 1 and 0, as BF16 pairs (2^-16 of a value) or in FP32
    assert bool(((xi - w.double()).abs() <= 2.0**-16 * w.double().abs()).all())
    m = 40
    C = torch.randn((n, m), generator=gen, dtype=torch.float64)
    out = torch.full((m, npts), 5.0, dtype=torch.float32, device="cuda")
    abi.ace_apply_finish(op, C.cuda(), out)
    # BF16 pairs: 2^-16 of the products' magnitudes; FP32 sums of three products per term, 2^-23 each
    bound = (2.0**-16 + (3 * n + 8) * 2.0**-23) * (C.T.abs() @ xi.abs())
    assert bool(((out.cpu().double() + C.T @ xi).abs() <= bound).all())
