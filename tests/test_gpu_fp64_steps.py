"""FP64 form: the Gram in small tiles and balanced chunks at the edges of its plan, and W from stored
potentials added in pack order, for every kind of pack, against the no-allocation route (atomic pencil
passes) and bit for bit against itself."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from gpu_helpers import FP64_ARRAY_RTOL, rel_max
from paper_2101_03155_gb300 import ace as abi
from workloads.generators import gaussian_orbitals

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 12, 16, 17, 32, 33, 64, 130])
@pytest.mark.parametrize("npts", [31, 64, 1000, 4097])
def test_gram_against_torch(n, npts):
    import torch

    gen = torch.Generator().manual_seed(1000 * n + npts)
    x = torch.randn((n, npts), generator=gen, dtype=torch.float64).cuda()
    y = torch.randn((n, npts), generator=gen, dtype=torch.float64).cuda()
    d = ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n, prec=ace.ACE_FP64)
    dV = 512.0 / 4096.0
    M = torch.empty((n, n), dtype=torch.float64, device="cuda")
    abi.ace_m_partial(d, x, y, M)
    ref = -dV * (x @ y.T)
    # 32-point partial sums, compensated sums over them, 8 interleaved sums over the chunks: under 100
    # roundings of 2^-53 on the sum of the products' magnitudes; torch's own sum has up to npts
    bound = (100 + npts) * 2.0**-53 * dV * (x.abs() @ y.abs().T)
    assert bool((torch.abs(M - ref) <= bound).all())


PAIRS = [[(0, 1)], [(2, 2)], [(0, 1), (0, 3)], [(1, 1), (4, 4)], [(0, 0), (0, 1)], [(0, 1), (2, 3)], [(0, 4), (2, 4)],
         [(i, j) for i in range(5) for j in range(i, 5)]]


@pytest.mark.parametrize("grid", [(6, 16, 16), (5, 15, 18), (12, 12, 24)])
@pytest.mark.parametrize("pairs", PAIRS)
def test_w_from_stored_potentials(grid, pairs):
    import torch

    lat = np.diag([6.0 + 0.05 * g for g in grid])
    phi, _, _ = gaussian_orbitals(grid, lat, 5, 2, np.random.default_rng(sum(grid)))
    x = torch.from_numpy(phi).cuda()
    d = ace.make_desc(grid, lat, 5, prec=ace.ACE_FP64)
    W = [torch.full_like(x, 7.0) for _ in range(3)]
    abi.ace_exchange_w(d, x, pairs, W[0])
    abi.ace_exchange_w(d, x, pairs, W[1])
    abi.ace_exchange_w_noalloc(d, x, pairs, W[2])
    torch.cuda.synchronize()
    assert torch.equal(W[0], W[1])
    assert rel_max(W[0].cpu().numpy(), W[2].cpu().numpy()) <= FP64_ARRAY_RTOL


@pytest.mark.parametrize("mb", ["1", "3", "64"])
def test_pencil_scratch_budget_leaves_w_alone(monkeypatch, mb):
    import torch

    grid = (5, 135, 81)  # a plane shape of the pencil route, 0.83 MB per pack
    lat = np.diag([6.0 + 0.05 * g for g in grid])
    phi, _, _ = gaussian_orbitals(grid, lat, 5, 2, np.random.default_rng(3))
    x = torch.from_numpy(phi).cuda()
    d = ace.make_desc(grid, lat, 5, prec=ace.ACE_FP64)
    W = [torch.full_like(x, 7.0) for _ in range(2)]
    abi.ace_exchange_w(d, x, PAIRS[-1], W[0])
    monkeypatch.setenv("ACE_SCRATCH_MB", mb)
    abi.ace_exchange_w(d, x, PAIRS[-1], W[1])
    torch.cuda.synchronize()
    assert torch.equal(W[0], W[1])
