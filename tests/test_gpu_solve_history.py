"""What a context solved before does not change what it solves next (the
number of CG steps that are queued ahead follows the last solve)."""

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_solves_do_not_depend_on_earlier_ones(lib, precision):
    """A solve after one that took many steps, after one of b = 0 (none) and
    after one from its own solution (none or few) is bitwise the same as on a
    fresh context."""
    g = (8, 8, 8)
    med = wl.chiral_sphere(g, 0.25, 13.0, 1.0, 0.5)
    rng = np.random.default_rng(3)
    n = 4 * 8 ** 3
    b = torch.from_numpy(rng.standard_normal(n) + 1j * rng.standard_normal(n)).cuda()

    def context():
        return lib.Context(g, (0.3, 0.2, 0.1), med, precision=precision, cg_tol=1e-11)

    with context() as c:
        x, info = c.cg_solve(b)
        assert info.iterations > 8
        again, _ = c.cg_solve(b)
        zero, zinfo = c.cg_solve(torch.zeros_like(b))
        assert zinfo.iterations == 0 and not torch.any(zero != 0)
        after_zero, _ = c.cg_solve(b)
        c.cg_solve(b, x0=x)
        after_start, info2 = c.cg_solve(b)
    for y in (again, after_zero, after_start):
        assert torch.equal(x, y)
    assert info2.iterations == info.iterations


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_eigensolves_repeat(lib, precision):
    g = (8, 8, 12)
    med = wl.chiral_sphere(g, 0.25, 13.0, 1.0, 0.5)
    with lib.Context(g, (0.3, 0.2, 0.1), med, precision=precision, cg_tol=1e-11, eig_tol=1e-10) as c:
        first, _, i1 = c.eigs(4, vectors=False)
        second, _, i2 = c.eigs(4, vectors=False)
    assert np.array_equal(first, second) and i1.cg_iterations == i2.cg_iterations
