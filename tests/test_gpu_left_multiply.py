"""Tensor-core left multiply and Gram pipelines at the edges of their tiles, rings and buffer plans
(1 to 9 row steps, one to several row blocks, fewer items than ring stages, ragged last tiles), against
FP64 sums."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from paper_2101_03155_gb300 import ace as abi

pytestmark = pytest.mark.gpu

# n: rows of xi (32 per step; three B buffers up to 160, two beyond, other kernel from 257 on);
# m: rows of the result (128 per block, 32 per output warp)
@pytest.mark.parametrize("npts", [32, 100, 128, 2592, 19456 * 3 + 36])
@pytest.mark.parametrize("n,m", [(9, 9), (16, 33), (32, 128), (33, 31), (96, 129), (128, 64), (160, 96), (161, 40),
                                 (256, 260), (257, 10)])
def test_coefficients_and_finish(n, m, npts):
    import torch

    gen = torch.Generator().manual_seed(97 * n + 13 * m + npts)
    w = torch.randn((n, npts), generator=gen, dtype=torch.float32).cuda()
    d = ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n)
    dV = 512.0 / 4096.0
    op = abi.ace_build_from_m(d, -torch.eye(n, dtype=torch.float64, device="cuda"), w)
    xi = torch.from_numpy(abi.get_numpy(op, abi.ACE_GET_XI).reshape(n, npts)).double()
    psi = torch.randn((m, npts), generator=gen, dtype=torch.float32)
    # BF16 pairs: each factor is off by at most 2^-18 of itself and the product of the two low parts,
    # left out, is at most 2^-18: under 2^-16 of the product of the magnitudes; the FP32 sums add at
    # most 2^-23 per addition (truncation), three products per term, over runs of at most 256 points
    # (Gram) or n terms (left multiply)
    C = torch.full((n, m), 3.0, dtype=torch.float64, device="cuda")
    abi.ace_apply_coeffs(op, psi.cuda(), C)
    p = psi.double()
    bound = (2.0**-16 + 3 * 260 * 2.0**-23) * dV * (xi.abs() @ p.abs().T)
    assert bool(((C.cpu() - dV * (xi @ p.T)).abs() <= bound).all())
    out = torch.full((m, npts), 5.0, dtype=torch.float32, device="cuda")
    abi.ace_apply_finish(op, C, out)
    A = C.cpu().T
    bound = (2.0**-16 + (3 * n + 8) * 2.0**-23) * (A.abs() @ xi.abs())
    assert bool(((out.cpu().double() + A @ xi).abs() <= bound).all())
