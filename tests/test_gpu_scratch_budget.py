"""ACE_SCRATCH_MB bounds the pair chain's scratch: the high-water mark of the device's memory pool follows it, on grids
of the line-pair planes and of the pencil passes, and W stays the same."""

import ctypes

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from gpu_helpers import MIXED_W_RTOL, rel_max
from paper_2101_03155_gb300 import ace as abi
from workloads.generators import gaussian_orbitals

pytestmark = pytest.mark.gpu

USED_HIGH = 8  # cudaMemPoolAttrUsedMemHigh


class _Pool:
    def __init__(self):
        abi.load()
        self.rt = ctypes.CDLL("libcudart.so.13")
        self.pool = ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.pool), 0) == 0

    def high_of(self, call):
        import torch

        torch.cuda.synchronize()
        v = ctypes.c_uint64(0)
        assert self.rt.cudaMemPoolSetAttribute(self.pool, USED_HIGH, ctypes.byref(v)) == 0
        call()
        torch.cuda.synchronize()
        assert self.rt.cudaMemPoolGetAttribute(self.pool, USED_HIGH, ctypes.byref(v)) == 0
        return v.value


@pytest.mark.parametrize("grid", [(40, 90, 100), (40, 80, 125)])  # 45 x 100 and 40 x 125: planes and pencils
@pytest.mark.parametrize("prec", [ace.ACE_MIXED, ace.ACE_FP64])
def test_budget_bounds_the_scratch(grid, prec, monkeypatch):
    import torch

    n = 12
    lat = np.diag([0.2 * g for g in grid])
    phi, _, _ = gaussian_orbitals(grid, lat, n, 1, np.random.default_rng(sum(grid)))
    fp64 = prec == ace.ACE_FP64
    x = torch.from_numpy(phi if fp64 else phi.astype(np.float32)).cuda()
    d = ace.make_desc(grid, lat, n, prec=prec)
    pairs = [(i, j) for i in range(n) for j in range(i, n)]
    pack = x[0].numel() * (16 if fp64 else 8)
    pool, W, high = _Pool(), {}, {}
    for mb in (200, 3 * pack // 2**20 + 1, 1):  # room for all streams, for three packs, for less than one
        monkeypatch.setenv("ACE_SCRATCH_MB", str(mb))
        W[mb] = torch.empty_like(x)
        abi.ace_exchange_w(d, x, pairs, W[mb])  # tables and pool ready
        high[mb] = pool.high_of(lambda: abi.ace_exchange_w(d, x, pairs, W[mb]))
    wide, three, one = high
    # the rest of the call's memory is the same: with one pack, its scratch and a little slack remain
    rest = high[one] - pack
    assert high[three] <= rest + three * 2**20 + 2**20
    assert high[wide] >= rest + 4 * pack
    monkeypatch.setenv("ACE_SCRATCH_MB", "0")  # no budget at all: one pack
    assert pool.high_of(lambda: abi.ace_exchange_w(d, x, pairs, W[one])) <= high[one] + 2**20
    for mb in (three, one):
        if fp64:
            assert torch.equal(W[mb], W[wide])
        else:
            assert rel_max(W[mb].cpu().numpy(), W[wide].cpu().numpy()) <= 2 * MIXED_W_RTOL


@pytest.mark.parametrize("prec", [ace.ACE_MIXED, ace.ACE_FP64])
def test_pencil_chain_has_64_mb_by_default(prec, monkeypatch):
    """A grid of pencil passes whose pack takes 20 MB (mixed) or 40 MB: three packs, or two in FP64."""
    import torch

    monkeypatch.delenv("ACE_SCRATCH_MB", raising=False)
    grid, n = (125, 125, 160), 4
    fp64 = prec == ace.ACE_FP64
    gen = torch.Generator(device="cuda").manual_seed(4)
    x = torch.rand((n,) + grid, generator=gen, device="cuda", dtype=torch.float64 if fp64 else torch.float32)
    d = ace.make_desc(grid, np.diag([10.0, 10.0, 12.0]), n, prec=prec)
    pairs = [(i, j) for i in range(n) for j in range(i, n)]
    W, pool = torch.empty_like(x), _Pool()
    abi.ace_exchange_w(d, x, pairs, W)
    high = pool.high_of(lambda: abi.ace_exchange_w(d, x, pairs, W))
    scratch = max(64 * 2**20, 2 * 16 * x[0].numel()) if fp64 else 64 * 2**20
    assert high <= x.numel() * x.element_size() + scratch + 4 * 2**20  # W, the scratch, small buffers
