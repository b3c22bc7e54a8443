"""The exact inner products of the orthogonality monitor: how long their FP32
sums run.  The rounding error of an FP32 sum grows with its length, so a thread's
sums may not be longer than those of one element at a time over all the blocks
that the library's reductions take (46 elements at 96^3, 64 at most in the
grids below)."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1402_6297_gb300 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("shim") / "exact_dots.so")
    subprocess.check_call([build.nvcc_path(), "-std=c++17", "-O3", "-shared", "-Xcompiler", "-fPIC"] + build.ARCH +
                          ["-I", build.CSRC, os.path.join(HERE, "shim", "exact_dots_shim.cu"), "-o", so])
    L = ctypes.CDLL(so)
    L.shim_exact_blocks.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    L.shim_red_blocks.argtypes = [ctypes.c_longlong, ctypes.c_int]
    vp = ctypes.c_void_p
    L.shim_exact_dots.argtypes = [vp, vp, vp, vp, ctypes.c_longlong, ctypes.c_int, ctypes.c_int, vp]
    return L


def run(shim, shi, slo, whi, wlo, P):
    m, N = shi.shape
    out = np.zeros((m, 2))
    assert shim.shim_exact_dots(shi.ctypes.data, slo.ctypes.data, whi.ctypes.data, wlo.ctypes.data, N, m, P,
                                out.ctypes.data) == 0
    return out[:, 0] + 1j * out[:, 1]


@pytest.mark.parametrize("edge,P", [(96, 1), (64, 1), (48, 16), (64, 4), (32, 16), (8, 3)])
@pytest.mark.parametrize("m", [3, 17])
def test_sums_of_the_small_terms(shim, edge, P, m):
    """1 + 2^-18 as the low part of every entry of w, ones as the basis: the
    multiples k (1 + 2^-18) are floats up to k = 64, so the result is exact
    while no FP32 sum is longer than that, and their sum (below 2^23, a multiple
    of 2^-18) is a double."""
    N = 4 * edge ** 3
    nb = shim.shim_red_blocks(N, P)
    assert -(-N // (256 * nb)) <= 64
    c = np.float32(1 + 2.0 ** -18)
    ones = np.ones((m, N), dtype=np.complex64)
    out = run(shim, ones, np.zeros_like(ones), np.zeros(N, np.complex64), np.full(N, c, dtype=np.complex64), P)
    assert np.array_equal(out, np.full(m, N * float(c) + 0j))


@pytest.mark.parametrize("edge,m", [(8, 1), (8, 16), (12, 15), (32, 33)])
def test_against_the_sum_in_64_bits(shim, edge, m):
    """Random vectors: within 2^-52 log2(N) of the sum of the terms' magnitudes,
    what the FP64 additions of the partials and of the reference may leave."""
    N = 4 * edge ** 3
    rng = np.random.default_rng(edge)
    S = rng.standard_normal((m, N)) + 1j * rng.standard_normal((m, N))
    w = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    parts = []
    for v in (S, w):
        hi = v.astype(np.complex64)
        parts += [hi, (v - hi).astype(np.complex64)]
    out = run(shim, *parts, P=1)
    scale = np.abs(S) @ np.abs(w)
    assert np.all(np.abs(out - S.conj() @ w) <= 2.0 ** -52 * scale * np.log2(N))
