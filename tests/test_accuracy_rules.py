"""Host rules that bound the rounding errors of the solver's kernels (no GPU):
called in the built library by their C++ names."""
import ctypes
import os
import struct
from fractions import Fraction

import numpy as np
import pytest

LIB = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_03148_gb300", "libcell.so")


@pytest.fixture(scope="module")
def lib():
    if not os.path.exists(LIB):
        from paper_2410_03148_gb300 import build
        build.build()
    return ctypes.CDLL(LIB)


def test_coarsest_inverse_is_kept_only_at_its_own_precision(lib):
    """Newton-Schulz leaves the square of the residual R before its last step,
    entries of at most n max|R|^2 with n <= 224 unknowns: an inverse is kept if
    that is below FP64 rounding (2^-52), or FP32 rounding (2^-24) where it is
    stored in FP32, and never with a residual that is no number."""
    failed = lib._ZN4cell19dense_invert_failedEjb
    failed.argtypes, failed.restype = (ctypes.c_uint, ctypes.c_bool), ctypes.c_bool
    bits = lambda v: struct.unpack("I", struct.pack("f", v))[0]
    for fp64, eps in ((True, 2.0 ** -52), (False, 2.0 ** -24)):
        edge = (eps / 224) ** 0.5
        assert failed(bits(1.01 * edge), fp64)
        assert failed(bits(float("nan")), fp64) and failed(bits(float("inf")), fp64)
        assert not failed(bits(0.2 * edge), fp64) and not failed(0, fp64)


def test_gram_schmidt_chains_are_short(lib):
    """A thread of the Gram-Schmidt dots chains FP32 products before its value
    enters the block's compensated sum: at most 32 until a load has 1024 blocks
    of 256 threads, the fewest blocks of a load's other reductions."""
    blocks = lib._ZN4cell9gs_blocksEx
    blocks.argtypes, blocks.restype = (ctypes.c_longlong,), ctypes.c_int
    for n in list(range(2, 130)) + [160, 192, 256, 400, 736]:
        length = 4 * n ** 3
        b = blocks(length)
        assert 1 <= b <= 1024
        assert b >= min(1024, -(-length // (32 * 256))), n


@pytest.mark.parametrize("nc", [1, 3, 4])
def test_modal_matrix_is_the_rounded_exact_transform(lib, nc):
    """H K H^T / 64 (H: sums and differences along the axes) of matrices whose
    entries span 30 binary orders, against exact rational arithmetic: every
    entry is the nearest double, whatever the host's long double is."""
    fn = lib._ZN8cellhost12modal_matrixEPKdiPd
    fn.argtypes, fn.restype = (ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p), None
    R = 8 * nc
    H = np.array([[np.prod([(1 if a >> b & 1 else -1) if m >> b & 1 else 1 for b in range(3)]) for a in range(8)] for m in range(8)])
    for seed in range(12 // nc):
        rng = np.random.default_rng(seed)
        K = rng.uniform(-1, 1, (R, R)) * 2.0 ** -rng.integers(0, 30, (R, R))
        got = np.empty((R, R))
        fn(K.ctypes.data, nc, got.ctypes.data)
        F = np.array([Fraction(v) for v in K.ravel()], dtype=object).reshape(8, nc, 8, nc)
        want = np.einsum("ma,acbd->mcbd", H.astype(object), F)
        want = np.einsum("nb,mcbd->mcnd", H.astype(object), want).reshape(R, R)
        assert all(g == float(w / 64) for g, w in zip(got.ravel(), want.ravel()))
