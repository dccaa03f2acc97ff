"""One-CTA Cholesky of up to 32 orbitals on matrices near the ends of the FP64 range, where a pivot's reciprocal
has no FP64 value: powers of four scale L and L^-1 exactly."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from paper_2101_03155_gb300 import ace as abi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 9, 32])
@pytest.mark.parametrize("exponent", [-1034, -1000, 1000])
def test_scaled(n, exponent):
    import torch

    B = np.random.default_rng(n).integers(-4, 5, (n, n)).astype(float)
    A = B @ B.T + 64.0 * np.eye(n)  # whole numbers below 2^11: the scaled entries are exact
    d = ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n, prec=ace.ACE_FP64)
    W = torch.eye(n, dtype=torch.float64, device="cuda")
    out = []
    for e in (0, exponent):
        op = abi.ace_build_from_m(d, torch.from_numpy(np.ldexp(-A, e)).cuda(), W)
        out.append((np.ldexp(abi.get_numpy(op, abi.ACE_GET_L), -e // 2),
                    np.ldexp(abi.get_numpy(op, abi.ACE_GET_XI).reshape(n, n), e // 2)))
    # the eliminated matrix has 2^-1074 for its last bit at the small end: 2^-40 of its entries, n updates
    # of each element, and a condition below 64
    tol = 64 * n * 2.0**-40 if exponent == -1034 else 64 * n * 2.0**-53
    for a, b in zip(*out):
        assert np.all(np.isfinite(b)) and np.abs(a - b).max() <= tol * np.abs(a).max()
