"""CUDA-core left multiply in FP64 at the edges of its row blocks, with a triangular factor (xi) and a full
one (the application), against torch."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from paper_2101_03155_gb300 import ace as abi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npts", [1, 63, 64, 1000])
@pytest.mark.parametrize("n,m", [(1, 1), (12, 16), (16, 17), (17, 33), (33, 64), (48, 65), (70, 12), (130, 140)])
def test_triangular_and_full_factor(n, m, npts):
    import torch

    gen = torch.Generator().manual_seed(n + m + npts)
    W = torch.randn((n, npts), generator=gen, dtype=torch.float64)
    B = torch.randn((n, n), generator=gen, dtype=torch.float64)
    M = -(B @ B.T + n * torch.eye(n, dtype=torch.float64))
    d = ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n, prec=ace.ACE_FP64)
    op = abi.ace_build_from_m(d, M.cuda(), W.cuda())
    L = torch.from_numpy(abi.get_numpy(op, abi.ACE_GET_L))
    xi = torch.from_numpy(abi.get_numpy(op, abi.ACE_GET_XI).reshape(n, npts))
    # L xi = W to the rounding of n-term sums, in the factor's inverse and in the product
    bound = 8 * (n + 2) * 2.0**-53 * float(torch.linalg.cond(L)) * (L.abs() @ xi.abs())
    assert bool(((L @ xi - W).abs() <= bound).all())
    C = torch.randn((n, m), generator=gen, dtype=torch.float64)
    out = torch.full((m, npts), 5.0, dtype=torch.float64, device="cuda")
    abi.ace_apply_finish(op, C.cuda(), out)
    bound = (n + 2) * 2.0**-53 * (C.T.abs() @ xi.abs()) * 2
    assert bool(((out.cpu() + C.T @ xi).abs() <= bound).all())
