"""The device GMRES behind the NFSEP eigensolve at vector lengths on both sides
of its dispatch (several groups of basis vectors per update below 152 * 4 warps
of elements, one above; overlapping launches below 152 * 256 elements), and the
batch after a truncated one.  Each returned pair is checked by its own residual
||M y - omega y|| / (|omega| ||y||) with the library's product, whose parity with
the oracle test_gpu_nfsep checks: eig_tol bounds the Ritz residual of the
inverse, so the residual here is within ||M - sigma|| / |omega - sigma| of it."""

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

K = (0.1, 0.2, 0.3)
SIGMA = 2.0 + 0.1j


@pytest.mark.parametrize("grid", [(8, 8, 8), (8, 8, 24), (12, 12, 12), (24, 24, 16)],
                         ids=lambda g: "x".join(map(str, g)))
def test_eigenpair_residual(lib, grid):
    med = wl.biisotropic_sphere(grid, 0.25, 13.0 + 2.0j, 1.0, 0.5, 0.2)
    ctx = lib.NFSEPContext(grid, K, med, cg_tol=1e-9, eig_tol=1e-6, cg_maxit=20000)
    omega, Y, info = ctx.eigs(1, SIGMA)
    assert info.nconv == 1
    y = Y[0].contiguous()
    My = ctx.matvec(y)
    res = float((My - complex(omega[0]) * y).norm() / (abs(omega[0]) * y.norm()))
    # ||M|| is at most the largest singular value of the curl, 2 sqrt(sum n_l^2)
    bound = (2.0 * np.sqrt(sum(n * n for n in grid)) + abs(SIGMA)) / abs(omega[0] - SIGMA) * 1e-6 * 10
    assert res < bound, (res, bound)


def test_iteration_cap_is_kept(lib):
    """maxit that is no multiple of the batch: the solve stops there, counted exactly."""
    grid = (8, 8, 8)
    med = wl.biisotropic_sphere(grid, 0.25, 13.0 + 2.0j, 1.0, 0.5, 0.2)
    ctx = lib.NFSEPContext(grid, K, med, cg_maxit=137)
    omega, _, info = ctx.eigs(1, SIGMA, allow_noconv=True)
    assert info.status == lib.NFS_ENOCONV and info.gmres_iterations == 137
    assert np.all(omega == 0)
