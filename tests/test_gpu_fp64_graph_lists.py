"""FP64 graphs on short pair lists, where fewer batches than side streams exist: the chain forks no stream
that it does not join (the idle ones of five packs on four streams get no work), and the replay equals
ace_build_pairs bit for bit."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from paper_2101_03155_gb300 import ace as abi
from workloads.generators import gaussian_orbitals

pytestmark = pytest.mark.gpu


def _list(npairs, n):
    """The n diagonal pairs first (the exchange matrix needs them), then the others."""
    every = [(i, i) for i in range(n)] + [(i, j) for i in range(n) for j in range(i + 1, n)]
    return np.array(sorted(every[:npairs]), dtype=np.int32)


@pytest.mark.parametrize("grid", [(12, 16, 16), (5, 15, 18)])
@pytest.mark.parametrize("n,npairs", [(1, 1), (2, 3), (3, 6), (4, 10), (5, 9), (6, 18), (6, 21)])
def test_short_lists(n, npairs, grid):
    import torch

    lat = np.diag([6.0 + 0.05 * g for g in grid])
    phi, _, _ = gaussian_orbitals(grid, lat, n, 1, np.random.default_rng(10 * n + npairs))
    x = torch.from_numpy(phi).cuda()
    d = ace.make_desc(grid, lat, n, prec=ace.ACE_FP64)
    stream = torch.cuda.current_stream()
    pairs = _list(npairs, n)
    with ace.ace_graph_create([d], [x], [pairs], stream) as g:
        g.launch(stream)
        g.sync()
        want = ace.ace_build_pairs(d, x, pairs, stream)
        for what in (abi.ACE_GET_W, abi.ACE_GET_XI):
            assert np.array_equal(abi.get_numpy(g.ops[0], what), abi.get_numpy(want, what))
        want.close()

