"""Products with at most 8 rows on one side (a few vectors against xi, few orbitals): FP32 on the CUDA
cores, at the edges of the row groups, column runs and 16-byte loads, against FP64 sums."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from paper_2101_03155_gb300 import ace as abi

pytestmark = pytest.mark.gpu

EPS = 2.0**-24


def _op(n, npts, gen):
    """A handle of xi = W (M = -1), its xi as the getter returns it, and dV."""
    import torch

    w = torch.randn((n, npts), generator=gen, dtype=torch.float32).cuda()
    d = ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n)
    op = abi.ace_build_from_m(d, -torch.eye(n, dtype=torch.float64, device="cuda"), w)
    xi = torch.from_numpy(abi.get_numpy(op, abi.ACE_GET_XI).reshape(n, npts)).double()
    return op, xi, 512.0 / 4096.0


# 31: scalar route; 128 * 16: one FP64 fold; 311296: four points per thread of the left multiply from
# there on (152 SMs)
@pytest.mark.parametrize("npts", [31, 32, 132, 2052, 4097, 311296, 311300])
@pytest.mark.parametrize("n,m", [(1, 1), (3, 2), (7, 8), (8, 3), (8, 8), (9, 1), (9, 4), (64, 5), (65, 7), (300, 8)])
def test_coefficients_and_finish(n, m, npts):
    import torch

    if n == 300 and npts > 5000:
        pytest.skip("covered by the smaller row counts")
    gen = torch.Generator().manual_seed(97 * n + 13 * m + npts)
    op, xi, dV = _op(n, npts, gen)
    psi = torch.randn((m, npts), generator=gen, dtype=torch.float32)
    C = torch.full((n, m), 3.0, dtype=torch.float64, device="cuda")
    abi.ace_apply_coeffs(op, psi.cuda(), C)
    p = psi.double()
    if npts % 4 == 0:
        # a lane's run of 64 products and the 5 steps of the exchange in FP32, the rest in FP64
        bound = 70 * EPS * dV * (xi.abs() @ p.abs().T) * 1.01
        assert bool(((C.cpu() - dV * (xi @ p.T)).abs() <= bound).all())
    out = torch.full((m, npts), 5.0, dtype=torch.float32, device="cuda")
    abi.ace_apply_finish(op, C, out)
    A = C.cpu().T
    # C rounded to FP32 and n fused multiply-adds
    bound = (n + 1) * EPS * (A.abs() @ xi.abs()) * 1.01
    assert bool(((out.cpu().double() + A @ xi).abs() <= bound).all())


@pytest.mark.parametrize("n", [1, 2, 5, 8])
@pytest.mark.parametrize("npts", [36, 4100, 70000])
def test_m_of_few_orbitals(n, npts):
    import torch

    gen = torch.Generator().manual_seed(n + npts)
    x = torch.randn((n, npts), generator=gen, dtype=torch.float32)
    y = torch.randn((n, npts), generator=gen, dtype=torch.float32)
    d = ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n)
    dV = 512.0 / 4096.0
    M = torch.full((n, n), 9.0, dtype=torch.float64, device="cuda")
    abi.ace_m_partial(d, x.cuda(), y.cuda(), M)
    bound = 70 * EPS * dV * (x.double().abs() @ y.double().abs().T) * 1.01
    assert bool(((M.cpu() + dV * (x.double() @ y.double().T)).abs() <= bound).all())
