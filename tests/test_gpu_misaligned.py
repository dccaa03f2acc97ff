"""Device arrays of the multi-GPU steps that start off a 16-byte boundary go through aligned copies: W of
ace_exchange_w (added in pairs of points) on every kind of grid, and the slabs of ace_m_partial (read in
16-byte vectors) on every route of the Gram."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from gpu_helpers import MIXED_W_RTOL, rel_max
from paper_2101_03155_gb300 import ace as abi
from workloads.generators import gaussian_orbitals

pytestmark = pytest.mark.gpu

OFFSETS = [1, 2, 3]  # in elements


def _shifted(t, off):
    """A copy of t that starts `off` elements past a 16-byte boundary."""
    import torch

    buf = torch.full((t.numel() + 4,), 7.0, dtype=t.dtype, device="cuda")
    v = buf[off:off + t.numel()].view(t.shape)
    v.copy_(t)
    assert v.is_contiguous() and buf.data_ptr() % 16 == 0
    return v, buf


@pytest.mark.parametrize("prec", [ace.ACE_MIXED, ace.ACE_FP64])
@pytest.mark.parametrize("grid", [(6, 16, 16), (5, 15, 18), (6, 12, 25), (8, 20, 45)])
@pytest.mark.parametrize("off", OFFSETS)
def test_exchange_w(prec, grid, off):
    import torch

    n = 5
    lat = np.diag([6.0 + 0.05 * g for g in grid])
    phi, _, _ = gaussian_orbitals(grid, lat, n, 2, np.random.default_rng(sum(grid)))
    x = torch.from_numpy(phi if prec == ace.ACE_FP64 else phi.astype(np.float32)).cuda()
    d = ace.make_desc(grid, lat, n, prec=prec)
    pairs = [(i, j) for i in range(n) for j in range(i, n)]
    want = torch.empty_like(x)
    abi.ace_exchange_w(d, x, pairs, want)
    got, buf = _shifted(torch.full_like(x, 3.0), off)
    abi.ace_exchange_w(d, _shifted(x, off)[0], pairs, got)
    torch.cuda.synchronize()
    assert rel_max(got.cpu().numpy(), want.cpu().numpy()) <= (2 * MIXED_W_RTOL if prec == ace.ACE_MIXED else 0.0)
    assert bool((buf[:off] == 7.0).all()) and bool((buf[off + x.numel():] == 7.0).all())


@pytest.mark.parametrize("prec", [ace.ACE_MIXED, ace.ACE_FP64])
@pytest.mark.parametrize("n,npts", [(4, 132), (12, 4096), (12, 100), (40, 4097), (130, 2048)])
@pytest.mark.parametrize("off", OFFSETS)
def test_m_partial(prec, n, npts, off, monkeypatch):
    import torch

    gen = torch.Generator().manual_seed(n + npts)
    dt = torch.float64 if prec == ace.ACE_FP64 else torch.float32
    x = torch.randn((n, npts), generator=gen, dtype=dt).cuda()
    y = torch.randn((n, npts), generator=gen, dtype=dt).cuda()
    d = ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n, prec=prec)
    for env in (None, "ACE_NO_TMA", "ACE_NO_TC"):
        if env:
            monkeypatch.setenv(env, "1")
        M = [torch.empty((n, n), dtype=torch.float64, device="cuda") for _ in range(2)]
        abi.ace_m_partial(d, x, y, M[0])
        abi.ace_m_partial(d, _shifted(x, off)[0], _shifted(y, off)[0], M[1])
        # the same kernels on the same values; FP64 atomics add the chunks of some routes in any order
        tol = 2.0**-45 * (x.double().abs() @ y.double().abs().T) / 8.0
        assert bool(((M[0] - M[1]).abs() <= tol).all())
        if env:
            monkeypatch.delenv(env)
