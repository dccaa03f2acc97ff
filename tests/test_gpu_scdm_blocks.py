"""The FP32 pivot selection on block bounds: point counts off the 8-point block and the 16-byte row, more
orbitals than one round of a warp holds, as many points as orbitals, and ties; every pivot must have the
largest residual norm to FP32 rounding, the first index winning exact ties."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from test_gpu_scdm import _check_pivots, _gpu_scdm

pytestmark = pytest.mark.gpu


def _smooth(n, grid, seed):
    """n random sums of plane waves and bumps on the grid (no symmetry, well separated residuals)."""
    rng = np.random.default_rng(seed)
    x = np.stack(np.meshgrid(*[np.arange(g) / g for g in grid], indexing="ij"), -1).reshape(-1, 3)
    c = rng.uniform(0, 1, (n, 3))
    d = x[None] - c[:, None]
    d -= np.round(d)
    bumps = np.exp(-(d**2).sum(-1) / (2 * rng.uniform(0.05, 0.2, (n, 1)) ** 2))
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    return (q @ (bumps + 1e-3 * rng.standard_normal(bumps.shape))).reshape((n,) + grid)


@pytest.mark.parametrize("n,grid", [(1, (2, 2, 2)), (6, (1, 2, 3)), (5, (7, 9, 11)), (31, (10, 10, 10)), (33, (9, 10, 12)),
                                    (128, (16, 18, 20)), (130, (16, 18, 20)), (160, (15, 15, 15)), (20, (48, 48, 48))])
def test_pivots_are_greedy(n, grid):
    psi = _smooth(n, grid, 100 * n + grid[2])
    g = _gpu_scdm(psi, ace.ACE_MIXED)
    assert g["status"] == 0, ace.ace_last_error()
    # 2e-5: the FP32 projections' error bound of the other selection tests
    _check_pivots(g["input"], g["piv"], 2e-5)
    assert np.abs(g["U"].T @ g["U"] - np.eye(n)).max() <= 1e-9


def test_exact_ties_take_the_first_index():
    psi = _smooth(4, (8, 8, 9), 5)
    twice = np.concatenate([psi, psi], axis=1)  # every column appears twice
    a = _gpu_scdm(psi, ace.ACE_MIXED)
    b = _gpu_scdm(twice, ace.ACE_MIXED)
    assert list(a["piv"]) == list(b["piv"])
