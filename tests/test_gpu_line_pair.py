"""The FP32 plane chain that transforms two lines per thread: plane shapes at the edges of its work split
(odd and even axes 2 and 3 in every combination, planes in groups of lines and whole-CTA planes, one
plane per SM), axis-1 lengths with short last tiles, and every kind of pack, against the FP64 oracle and
the five pencil passes."""

import numpy as np
import pytest

import oracle
import paper_2101_03155_gb300 as ace
from gpu_helpers import MIXED_W_RTOL, gpu_build, rel_max
from paper_2101_03155_gb300 import ace as abi
from workloads.generators import gaussian_orbitals

pytestmark = pytest.mark.gpu


def _orbitals(grid, n, seed):
    lat = np.diag([6.0 + 0.05 * g for g in grid])
    phi, _, _ = gaussian_orbitals(grid, lat, n, 2, np.random.default_rng(seed))
    return phi, lat


# axis 2 x axis 3: even x odd, odd x even, odd x odd, even x even; small planes (warp or 64-thread groups
# of lines), planes above 64 x 64 (whole CTA), planes of which one fills an SM; axis 1 from 2 to 256
GRIDS = [(2, 24, 25), (3, 25, 24), (5, 27, 27), (16, 12, 24), (256, 16, 12), (9, 32, 48), (6, 45, 50), (4, 50, 45),
         (10, 75, 80), (4, 80, 75), (3, 81, 81), (2, 135, 128), (2, 128, 135), (2, 160, 144), (5, 15, 18)]


@pytest.mark.parametrize("grid", GRIDS)
def test_plane_shapes_against_the_oracle(grid):
    phi, lat = _orbitals(grid, 4, sum(grid) + 3)
    ref = oracle.ace_build(phi, lat, 0.0, 2.0)
    g = gpu_build(phi, lat, ace.ACE_MIXED)
    assert g["status"] == 0
    assert rel_max(g["W"].reshape(ref["W"].shape), ref["W"]) <= MIXED_W_RTOL


# one pair, a diagonal pair, two pairs sharing an orbital, two diagonal pairs, a diagonal and an
# off-diagonal pair of one orbital, two pairs without a common orbital, and a longer mixed list
PAIRS = [[(0, 1)], [(2, 2)], [(0, 1), (0, 3)], [(1, 1), (4, 4)], [(0, 0), (0, 1)], [(0, 1), (2, 3)],
         [(0, 0), (0, 4), (1, 2), (1, 3), (2, 2), (3, 4), (4, 4)]]


@pytest.mark.parametrize("grid", [(6, 32, 32), (5, 27, 25), (4, 75, 72), (3, 96, 100)])
@pytest.mark.parametrize("pairs", PAIRS)
def test_packs_against_the_pencil_passes(grid, pairs, monkeypatch):
    import torch

    phi, lat = _orbitals(grid, 5, sum(grid))
    x = torch.from_numpy(phi.astype(np.float32)).cuda()
    d = ace.make_desc(grid, lat, 5, prec=ace.ACE_MIXED)
    out = []
    for pencil in ("0", "1"):
        monkeypatch.setenv("ACE_FORCE_PENCIL", pencil)
        W = torch.full_like(x, 7.0)
        abi.ace_exchange_w(d, x, pairs, W)
        out.append(W.cpu().numpy())
    touched = sorted({i for p in pairs for i in p})
    # rounding of the two FP32 routes, MIXED_W_RTOL each
    assert rel_max(out[0], out[1]) <= 2 * MIXED_W_RTOL
    rest = [i for i in range(5) if i not in touched]
    assert np.all(out[0][rest] == 0.0)
