"""Sums over the K-splits of the tensor-core Gram: as many bits as FP64, on inputs whose products and sums inside a
split are exact, and beyond the range of FP32."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace
from paper_2101_03155_gb300 import ace as abi

pytestmark = pytest.mark.gpu


def _m(n, x, y):
    import torch

    d = ace.make_desc((16, 16, 16), np.diag([8.0, 8.0, 8.0]), n)  # dV = 1/8
    M = torch.empty((n, n), dtype=torch.float64, device="cuda")
    abi.ace_m_partial(d, x.cuda(), y.cuda(), M)
    return M.cpu()


@pytest.mark.parametrize("n", [16, 130])
def test_sum_keeps_53_bits(n):
    """Three products of 2^30, 2^4 and 2^-22 in K-steps that the same slice of the splits adds up."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    splits = max(1, sms // (-(-n // 128)) ** 2)  # one tile of 128 x 128 per block pair
    npts = 256 * splits
    x = torch.zeros((n, npts))
    want = 0.0
    for k, e in ((0, 15), (16, 2), (32, -11)):
        assert k < splits
        x[:, 32 * k] = 2.0**e
        want += 4.0**e
    assert torch.equal(_m(n, x, x), torch.full((n, n), -want / 8.0, dtype=torch.float64))


def test_sum_beyond_fp32():
    """Two splits of 2^127 each: their sum has no FP32 value."""
    import torch

    n, npts = 16, 256 * torch.cuda.get_device_properties(0).multi_processor_count
    x = torch.zeros((n, npts))
    y = torch.zeros((n, npts))
    x[:, 0] = x[:, 512] = 2.0**63
    y[:, 0] = y[:, 512] = 2.0**64
    assert torch.equal(_m(n, x, y), torch.full((n, n), -(2.0**125), dtype=torch.float64))
