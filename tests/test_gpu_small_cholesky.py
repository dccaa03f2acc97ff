"""One-CTA Cholesky of up to 32 orbitals at the edges of its column slots and lanes, against LAPACK, and its
status codes."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from paper_2101_03155_gb300 import ace as abi

pytestmark = pytest.mark.gpu


def _desc(n):
    return ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n, prec=ace.ACE_FP64)


def _build(n, M, check=True):
    import torch

    W = torch.eye(n, dtype=torch.float64, device="cuda")
    return abi.ace_build_from_m(_desc(n), torch.from_numpy(np.ascontiguousarray(M)).cuda(), W, check=check)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 24, 25, 31, 32, 33])
def test_factor_and_inverse(n):
    rng = np.random.default_rng(n)
    B = rng.standard_normal((n, n))
    A = B @ B.T + 0.1 * n * np.eye(n)
    skew = rng.standard_normal((n, n)) * 1e-3
    op = _build(n, -(A + skew - skew.T))  # the antisymmetric part drops out
    L = abi.get_numpy(op, abi.ACE_GET_L)
    ref = np.linalg.cholesky(A)
    cond = np.linalg.cond(A)
    # backward error of the elimination and of the symmetrised input, n roundings each, times the condition
    tol = 8 * (n + 2) * cond * 2.0**-53
    assert np.abs(L - ref).max() <= tol * np.abs(ref).max()
    assert np.all(np.triu(L, 1) == 0.0)
    X = abi.get_numpy(op, abi.ACE_GET_XI).reshape(n, n)  # L^-1, since W = 1
    assert np.all(np.triu(X, 1) == 0.0)
    inv = np.linalg.inv(ref)
    assert np.abs(X - inv).max() <= tol * np.abs(inv).max()
    assert abs(ace.exchange_energy(op) + np.trace(A) * _desc(n).spin_factor / 2) <= 1e-14 * n * np.trace(A)


@pytest.mark.parametrize("n,j", [(1, 0), (8, 7), (9, 8), (16, 0), (24, 17), (32, 31)])
@pytest.mark.parametrize("pivot", [0.0, -1.0])
def test_failed_pivot(n, j, pivot):
    A = np.eye(n)
    A[j, j] = pivot
    st, _ = _build(n, -A, check=False)
    assert st == abi.ACE_ERR_NOT_POSDEF


@pytest.mark.parametrize("n", [1, 16, 32])
def test_non_finite_entry(n):
    A = np.eye(n)
    A[n - 1, 0] = np.nan
    st, _ = _build(n, -A, check=False)
    assert st == abi.ACE_ERR_NONFINITE
