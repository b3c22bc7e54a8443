"""How many CG steps are queued before the host looks."""

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_a_long_solve_from_a_bad_start_queues_nothing_for_later_ones(lib, precision):
    """A start 1e10 times too large takes many more steps than a solve from zero:
    an eigensolve after it launches the same kernels as on a fresh context (steps
    queued past convergence do nothing, but take their launches' time)."""
    g = (8, 8, 8)
    rng = np.random.default_rng(3)
    n = 4 * 8 ** 3

    def vec():
        return torch.from_numpy(rng.standard_normal(n) + 1j * rng.standard_normal(n)).cuda()

    def context():
        return lib.Context(g, (0.3, 0.2, 0.1), wl.chiral_sphere(g, 0.25, 13.0, 1.0, 0.5), precision=precision,
                           cg_tol=1e-11)

    with context() as c:
        omega, _, fresh = c.eigs(4, vectors=False)
    with context() as c:
        steps = c.cg_solve(vec())[1].iterations
        with_start = c.cg_solve(vec(), x0=1e10 * vec())[1]
    assert with_start.status == lib.NFS_OK and with_start.iterations > steps + 16
    with context() as c:
        c.cg_solve(vec(), x0=1e10 * vec())
        again, _, info = c.eigs(4, vectors=False)
    assert np.array_equal(omega, again)
    assert info.kernel_launches == fresh.kernel_launches
