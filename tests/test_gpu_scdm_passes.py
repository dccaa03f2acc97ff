"""The ways through the FP32 pivot selection (passes over every point, steps over block bounds, and the change from
these to passes over a point-major copy after any step) do the same arithmetic: the same pivots and U, on
orbitals that localise and on plane waves that do not, and on point counts off every tile."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from test_gpu_scdm import _check_pivots, _gpu_scdm
from test_gpu_scdm_blocks import _smooth

pytestmark = pytest.mark.gpu


def _waves(n, grid, seed):
    """Plane waves of the smallest wave vectors, rotated among each other: |psi(r)|^2 is almost constant."""
    rng = np.random.default_rng(seed)
    x = np.stack(np.meshgrid(*[np.arange(g) / g for g in grid], indexing="ij"), -1).reshape(-1, 3)
    k = sorted(((a * a + b * b + c * c, a, b, c) for a in range(-4, 5) for b in range(-4, 5) for c in range(-4, 5)))
    waves = [f(2 * np.pi * (x @ np.array(v[1:]))) for v in k[::2] for f in (np.cos, np.sin)]
    q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    psi = q @ np.array(waves[2:2 + n]) + 1e-3 * rng.standard_normal((n, x.shape[0]))
    return psi.reshape((n,) + grid)


@pytest.mark.parametrize("kind", [_smooth, _waves])
@pytest.mark.parametrize("n,grid", [(2, (3, 4, 5)), (9, (7, 9, 11)), (33, (9, 10, 12)), (70, (16, 18, 20)), (128, (15, 16, 17)),
                                    (131, (15, 15, 15)), (24, (48, 48, 45))])
def test_same_pivots(kind, n, grid, monkeypatch):
    psi = kind(n, grid, 10 * n + grid[2])
    want = _gpu_scdm(psi, ace.ACE_MIXED)
    assert want["status"] == 0, ace.ace_last_error()
    _check_pivots(want["input"], want["piv"], 2e-5)
    monkeypatch.setenv("ACE_SCDM_BOUNDS_MB", "0")
    for step in {0, 1, 2, n // 2, n - 2, n - 1}:
        monkeypatch.setenv("ACE_SCDM_LEAVE_STEP", str(max(step, 0)))
        got = _gpu_scdm(psi, ace.ACE_MIXED)
        assert got["status"] == 0, (step, ace.ace_last_error())
        assert list(got["piv"]) == list(want["piv"]), step
        assert np.array_equal(got["U"], want["U"]), step
