"""The kernels around a run of CG steps.  Its start: r^* r in float pairs.  The
end of a chunk: what the host is told where the sum that
stopped the steps and the check's own sum of the same partials round to the two
sides of the threshold.  A state that steps no more has to be reported as done,
or the host would queue chunks that do nothing for ever."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1402_6297_gb300 import build

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("shim") / "cg_check.so")
    subprocess.check_call([build.nvcc_path(), "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC"] + build.ARCH +
                          ["-I", build.CSRC, os.path.join(HERE, "shim", "cg_check_shim.cu"), "-o", so])
    return ctypes.CDLL(so)


@pytest.fixture(scope="module")
def shim(library):
    f = library.shim_cg_check
    d, i = ctypes.c_double, ctypes.c_int
    f.argtypes = [i, d, ctypes.POINTER(d), i, d, i, i, i, i, ctypes.POINTER(i), ctypes.POINTER(d)]

    def check(single, rr_now, part_b, tol2, halt, broken=0, it=5, maxit=100):
        part = np.ascontiguousarray(part_b, dtype=np.float64)
        out, rr = (i * 2)(), d()
        assert f(single, rr_now, part.ctypes.data_as(ctypes.POINTER(d)), part.size, tol2, halt, broken, it, maxit,
                 out, ctypes.byref(rr)) == 0
        return out[0], out[1], rr.value
    return check


@pytest.mark.parametrize("single", [0, 1])
def test_a_stopped_state_is_done(shim, single):
    tol2 = 1.0
    above = 1.0 + (2.0 ** -45 if single else 2.0 ** -52)
    # stopped by a sum at the threshold; the partials add up to just above it here
    assert shim(single, tol2, [0.5, above - 0.5], tol2, halt=1) == (1, 0, tol2)
    # still stepping: the partials decide
    assert shim(single, tol2, [0.5, above - 0.5], tol2, halt=0)[:2] == (0, 0)
    assert shim(single, 4.0, [0.5, 0.25], tol2, halt=0) == (1, 0, 0.75)
    # out of steps, and a breakdown
    assert shim(single, 4.0, [4.0], tol2, halt=1, it=100)[:2] == (1, -6)
    assert shim(single, 4.0, [4.0], tol2, halt=0, it=100)[:2] == (1, -6)
    assert shim(single, 4.0, [4.0], tol2, halt=1, broken=1)[:2] == (1, -7)
    assert shim(single, float("nan"), [float("nan")], tol2, halt=1)[:2] == (1, -7)


@pytest.mark.parametrize("n,nb", [(2, 1), (1024, 2), (65536, 19), (262144, 304)])
def test_start_of_an_inner_solve(library, n, nb):
    """Entries 1 and 2^-13 in turn: r^* r = n / 2 (1 + 2^-26), which a float pair
    holds (and every partial of it, of up to 2^7 elements a thread); an FP32 sum
    of both would drop the smaller square."""
    f = library.shim_inner_start
    f.argtypes = [ctypes.c_void_p, ctypes.c_longlong, ctypes.c_double, ctypes.c_int, ctypes.POINTER(ctypes.c_double)]
    r = np.zeros(n, dtype=np.complex128)
    r[0::2], r[1::2] = 0.5, 2.0 ** -14
    rr = ctypes.c_double()
    assert f(r.ctypes.data, n, 2.0, nb, ctypes.byref(rr)) == 0
    assert rr.value == n / 2 * (1 + 2.0 ** -26)
