"""FP32 Gram and left multiply on point counts off the 16-byte grid (the general kernels): edges of their tiles of
16, 32 and 64 rows, one and several chunks of points, and a triangular factor, against FP64 sums."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from paper_2101_03155_gb300 import ace as abi

pytestmark = pytest.mark.gpu

EPS = 2.0**-24
ROWS = [1, 9, 16, 17, 33, 64, 65, 97, 130, 200, 260]
POINTS = [31, 4097, 30011]


def _desc(n):
    return ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n)  # dV = 1/8


# 32 products in a row, a compensated sum of those (2 roundings) and the result's own, FP64 beyond 4096 points
GRAM = 36 * EPS


@pytest.mark.parametrize("n", ROWS)
@pytest.mark.parametrize("npts", POINTS)
def test_m(n, npts):
    import torch

    gen = torch.Generator().manual_seed(n + npts)
    x = torch.randn((n, npts), generator=gen, dtype=torch.float32)
    y = torch.randn((n, npts), generator=gen, dtype=torch.float32)
    M = torch.full((n, n), 9.0, dtype=torch.float64, device="cuda")
    abi.ace_m_partial(_desc(n), x.cuda(), y.cuda(), M)
    bound = GRAM / 8.0 * (x.double().abs() @ y.double().abs().T)
    assert bool(((M.cpu() + x.double() @ y.double().T / 8.0).abs() <= bound).all())


@pytest.mark.parametrize("n,m", [(9, 1), (17, 8), (33, 65), (65, 33), (130, 16), (200, 130)])
@pytest.mark.parametrize("npts", POINTS)
def test_coefficients(n, m, npts):
    import torch

    gen = torch.Generator().manual_seed(n + m + npts)
    w = torch.randn((n, npts), generator=gen, dtype=torch.float32)
    op = abi.ace_build_from_m(_desc(n), -torch.eye(n, dtype=torch.float64, device="cuda"), w.cuda())
    xi = torch.from_numpy(abi.get_numpy(op, abi.ACE_GET_XI).reshape(n, npts)).double()
    assert torch.equal(xi, w.double())  # the factor is one
    psi = torch.randn((m, npts), generator=gen, dtype=torch.float32)
    C = torch.full((n, m), 3.0, dtype=torch.float64, device="cuda")
    abi.ace_apply_coeffs(op, psi.cuda(), C)
    p = psi.double()
    assert bool(((C.cpu() - xi @ p.T / 8.0).abs() <= GRAM / 8.0 * (xi.abs() @ p.abs().T)).all())
    out = torch.full((m, npts), 5.0, dtype=torch.float32, device="cuda")
    abi.ace_apply_finish(op, C, out)
    A = C.cpu().T
    # C rounded to FP32 and n fused multiply-adds
    assert bool(((out.cpu().double() + A @ xi).abs() <= (n + 1) * 1.01 * EPS * (A.abs() @ xi.abs())).all())


@pytest.mark.parametrize("n", ROWS)
@pytest.mark.parametrize("npts", [31, 30011])
def test_xi(n, npts):
    import torch

    rng = np.random.default_rng(n)
    B = rng.standard_normal((n, n))
    A = B @ B.T + n * np.eye(n)
    w = torch.from_numpy(rng.standard_normal((n, npts)).astype(np.float32))
    op = abi.ace_build_from_m(_desc(n), torch.from_numpy(-A).cuda(), w.cuda())
    xi = torch.from_numpy(abi.get_numpy(op, abi.ACE_GET_XI).reshape(n, npts)).double()
    Li = torch.from_numpy(np.linalg.inv(abi.get_numpy(op, abi.ACE_GET_L)))
    # the factor rounded to FP32, n fused multiply-adds, and the FP64 inverse's own error far below
    bound = (n + 2) * EPS * (Li.abs() @ w.double().abs())
    assert bool(((xi - Li @ w.double()).abs() <= bound).all())
