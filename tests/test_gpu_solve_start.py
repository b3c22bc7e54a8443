"""Mixed-precision solves from a starting vector that is not zero."""

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("grid", [(8, 8, 8), (12, 12, 16), (32, 32, 24)])
@pytest.mark.parametrize("start", ["large", "random", "near"])
def test_residual_from_any_start(lib, grid, start):
    """The residual of the result, by the complex128 product, is within the
    tolerance: 1e-11 of |b|, and as much again for the rounding of the
    double-single residuals (1e-14 of |A_r| |x|, at most 1e3 |b| here)."""
    med = wl.chiral_sphere(grid, 0.25, 13.0, 1.0, 0.5)
    rng = np.random.default_rng(7)
    n = 4 * grid[0] * grid[1] * grid[2]

    def vec():
        return torch.from_numpy(rng.standard_normal(n) + 1j * rng.standard_normal(n)).cuda()

    with lib.Context(grid, (0.3, 0.2, 0.1), med, precision="mixed", cg_tol=1e-11) as c:
        b = vec()
        x0 = {"large": 1e4 * vec(), "random": vec(), "near": None}[start]
        if x0 is None:
            x0 = c.cg_solve(b)[0]
            x0 = x0 + 1e-9 * torch.linalg.norm(x0) * vec() / n ** 0.5
        x, info = c.cg_solve(b, x0=x0)
    with lib.Context(grid, (0.3, 0.2, 0.1), med, precision="fp64") as c:
        r = b - c.matvec(x)
    assert torch.linalg.norm(r) < 2e-11 * torch.linalg.norm(b)
    assert info.status == lib.NFS_OK
