"""The FP32 pivot selection on orbitals of very different norms: a residual keeps its own precision, however
small it is against the largest one."""

import numpy as np
import pytest

import paper_2101_03155_gb300 as ace

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [1, 10, 20, 40, 60])
def test_small_orbital_beside_a_large_one(exponent):
    """Orbital 0 is one on the first half of the grid, orbital 1 is 2^-exponent times a function on the second:
    the first pivot takes orbital 0 out exactly, the second one is the largest of two values of orbital 1
    whose squares differ by 2^-22."""
    import torch

    psi = np.zeros((2, 2, 8, 8), dtype=np.float32)
    psi[0, 0] = 1.0
    tail = np.full(64, 0.25, dtype=np.float32)
    tail[6], tail[37] = 1.0, 1.0 + 2.0**-23
    psi[1, 1] = (tail * np.float32(2.0**-exponent)).reshape(8, 8)
    x = torch.from_numpy(psi).cuda()
    # the status may say that the two columns are too unequal for their inverse square root
    _, piv, _, _ = ace.ace_scdm(x, torch.empty_like(x), ace.ACE_MIXED, torch.cuda.current_stream(), check=False)
    assert piv[0] == 0 and piv[1] == 64 + 37
