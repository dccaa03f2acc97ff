"""Residual norms of the FP32 SCDM selection (csrc/residual_key.h, plain C++ as well as device code): a key
holds its value exactly, keys compare like values, and an update v - p^2 is off by no more than an FP64
multiply-add may be (2^-53 of the result), against exact rational arithmetic."""

import ctypes
import os
import struct
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2101_03155_gb300", "csrc")
FRAC, BIAS, INF, NONE = 54, 383, 511 << 54, -(2**63)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("residual")
    src, so = d / "k.cpp", d / "k.so"
    src.write_text('#include "residual_key.h"\nextern "C" long long of_bits(unsigned b) { return ace::key_of_bits(b); }\n'
                   'extern "C" long long down(long long v, unsigned p) { return ace::key_downdate(v, p); }\n'
                   'extern "C" long long down_all(long long v, const unsigned *p, int n) {\n'
                   '  ace::KeySquare s[8];\n  for (int q = 0; q < 8; ++q) s[q] = ace::key_square(p[q]);\n'
                   '  return ace::key_close(ace::key_less_all<8>(ace::key_open(v), s, n), v); }\n'
                   'extern "C" long long below(long long v) { return ace::key_somewhat_below(v); }\n')
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(so), str(src)], check=True)
    k = ctypes.CDLL(str(so))
    k.of_bits.argtypes, k.of_bits.restype = [ctypes.c_uint32], ctypes.c_longlong
    k.down.argtypes, k.down.restype = [ctypes.c_longlong, ctypes.c_uint32], ctypes.c_longlong
    k.down_all.argtypes = [ctypes.c_longlong, ctypes.POINTER(ctypes.c_uint32), ctypes.c_int]
    k.down_all.restype = ctypes.c_longlong
    k.below.argtypes, k.below.restype = [ctypes.c_longlong], ctypes.c_longlong
    return k


def _bits(x):
    return struct.unpack("<I", struct.pack("<f", x))[0]


def _float(b):
    return struct.unpack("<f", struct.pack("<I", b))[0]


def _value(key):
    if key == 0:
        return Fraction(0)
    return Fraction((key & (1 << FRAC) - 1) | 1 << FRAC) * Fraction(2) ** ((key >> FRAC) - BIAS - FRAC)


EDGES = [0, 1, 2, 3, 0x7FFFFF, 0x800000, 0x800001, 0x3F800000, 0x3F7FFFFF, 0x3F800001, 0x7F7FFFFF]


def test_keys_of_norms(lib):
    rng = np.random.default_rng(1)
    bits = sorted(EDGES + [int(b) for b in rng.integers(0, 0x7F800000, 2000)])
    keys = [lib.of_bits(b) for b in bits]
    for b, k in zip(bits, keys):
        assert _value(k) == Fraction(_float(b))
    for a, b, ka, kb in zip(bits, bits[1:], keys, keys[1:]):
        assert (a < b) == (ka < kb)
    assert lib.of_bits(0x7F800000) == INF > max(keys)
    assert lib.of_bits(0x7FC00000) == lib.of_bits(0xFFC00000) == NONE


def _check(lib, v, p):
    """One update against v - p^2; the error bound is FP64's on the same operands."""
    r = lib.down(v, p)
    exact = _value(v) - Fraction(_float(p)) ** 2
    if exact <= 0:
        assert r == 0, (v, p)
    else:
        assert 0 <= _value(r) - exact <= Fraction(1, 2**53) * exact, (v, p)
    return r


def test_updates(lib):
    rng = np.random.default_rng(2)
    for b in EDGES:
        for p in EDGES:
            _check(lib, lib.of_bits(b), p)
            _check(lib, lib.of_bits(b), p | 0x80000000)
    for _ in range(3000):
        v = lib.of_bits(int(rng.integers(1, 0x7F800000)))
        while v > 0:  # a chain of updates by projections of up to the residual's size
            root = float(_value(v)) ** 0.5
            p = np.float32(min(root * 2.0 ** -rng.integers(0, 30) * rng.uniform(0.2, 1.0), 3e38))
            if rng.random() < 0.3:
                p = np.float32(min(root, 3e38))  # cancels to rounding
            w = _check(lib, v, _bits(float(p)))
            if w == v or rng.random() < 0.05:
                break
            v = w


def test_marks(lib):
    for p in EDGES + [0x7F800000, 0x7FC00000]:
        assert lib.down(-1, p) == -1 and lib.down(NONE, p) == NONE and lib.down(0, p) == 0
    one = lib.of_bits(0x3F800000)
    for p in (0x7F800000, 0xFF800000, 0x7FC00000):
        assert lib.down(one, p) == 0 and lib.down(INF, p) == 0
    assert lib.down(INF, 0x7F7FFFFF) == INF


def test_runs_equal_single_updates(lib):
    """Eight updates at once give the bits of eight updates in turn, whether the leading bit stays or moves."""
    rng = np.random.default_rng(4)
    special = [lib.of_bits(b) for b in EDGES] + [-1, NONE, INF]
    for trial in range(6000):
        v = special[trial % len(special)] if trial < 300 else lib.of_bits(int(rng.integers(1, 0x7F800000)))
        for _ in range(4):
            root = float(_value(v)) ** 0.5 if 0 < v < INF else 1.0
            scale = 2.0 ** -rng.integers(0, 40, 8) * rng.uniform(0, 1, 8) * rng.choice([1.0, 0.3, 0.02, 1.5])
            p = np.minimum(root * scale, 3e38).astype(np.float32)
            if rng.random() < 0.1:
                p[rng.integers(0, 8)] = rng.choice(np.array([0, np.inf, np.nan, 1e-45, 3e38], dtype=np.float32))
            bits = p.view(np.uint32)
            n = int(rng.integers(0, 9))
            want = v
            for q in range(n):
                want = lib.down(want, int(bits[q]))
            assert lib.down_all(v, (ctypes.c_uint32 * 8)(*[int(b) for b in bits]), n) == want
            if want <= 0:
                break
            v = want


def test_look_ahead_mark(lib):
    rng = np.random.default_rng(3)
    for b in rng.integers(0x800000, 0x7F800000, 500):
        v = lib.of_bits(int(b))
        q = _value(lib.below(v)) / _value(v)
        assert 0.66 < q < 0.85
    assert lib.below(0) == 0
