"""Solves that are given their own solution as the start."""

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GRIDS = [(8, 8, 8), (12, 12, 16), (32, 32, 24)]


def problem(lib, grid, precision):
    med = wl.chiral_sphere(grid, 0.25, 13.0, 1.0, 0.5)
    return lib.Context(grid, (0.3, 0.2, 0.1), med, precision=precision, cg_tol=1e-12)


def random_vector(grid, seed):
    rng = np.random.default_rng(seed)
    n = 4 * grid[0] * grid[1] * grid[2]
    return torch.from_numpy(rng.standard_normal(n) + 1j * rng.standard_normal(n)).cuda()


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("grid", GRIDS)
def test_the_solution_is_recognised_by_the_complex128_product(lib, grid, precision):
    """b = A_r x by the complex128 product: the residual of the start x, by the
    same product, is exactly zero.  (A residual of 48 bits leaves 1e-14 of
    |A_r| |x|, by which it would judge, and change, a better start.)"""
    with problem(lib, grid, precision) as c:
        x = random_vector(grid, 7)
        b = c.matvec(x)
        y, info = c.cg_solve(b, x0=x)
    assert torch.equal(x, y)
    assert (info.status, info.iterations, info.refinements, info.rel_residual) == (lib.NFS_OK, 0, 0, 0.0)


@pytest.mark.parametrize("where", [0, 1, 255, 256, -2, -1])
@pytest.mark.parametrize("grid", GRIDS)
def test_one_entry_makes_a_start(lib, grid, where):
    """A start with a single entry, however small, is not taken for a zero one."""
    with problem(lib, grid, "mixed") as c:
        x = torch.zeros_like(random_vector(grid, 7))
        x[where] = complex(0.0, 1e-120) if where % 2 else complex(-1e-120, 0.0)
        b = c.matvec(x)
        y, info = c.cg_solve(b, x0=x)
        assert torch.equal(x, y) and info.iterations == 0 and info.rel_residual == 0.0
        x[where] = complex(0.0, float("nan"))
        with pytest.raises(lib.NFSError):
            c.cg_solve(random_vector(grid, 8), x0=x)


@pytest.mark.parametrize("grid", GRIDS)
def test_a_zero_start_is_no_start(lib, grid):
    with problem(lib, grid, "mixed") as c:
        b = random_vector(grid, 9)
        x, info = c.cg_solve(b)
        y, again = c.cg_solve(b, x0=-torch.zeros_like(b))
    assert torch.equal(x, y) and info.iterations == again.iterations > 0
