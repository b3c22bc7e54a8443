"""The split of an eigensolve's time."""

import pytest

import workloads as wl

pytestmark = pytest.mark.gpu


def test_cg_seconds_do_not_hold_the_products_of_restarts(lib):
    """A basis of nev + 2 vectors restarts after every step and forms A_r V of
    12 vectors each time, about as many products as the step's CG takes
    (loose tolerance): a CG iteration still takes what it does without restarts,
    within a third for the few other kernels and the clock."""
    g = (48, 48, 48)
    per_iteration = {}
    for ncv, restarts in ((12, 12), (24, 0)):
        with lib.Context(g, (0.3, 0.2, 0.1), wl.chiral_sphere(g, 0.25, 13.0, 1.0, 0.5), precision="fp64", cg_tol=1e-4,
                         ncv=ncv, max_restarts=restarts) as c:
            c.eigs(10, vectors=False, allow_noconv=True)  # (the first one captures graphs)
            _, _, info = c.eigs(10, vectors=False, allow_noconv=True)
            assert info.restarts == restarts and info.cg_iterations > 24
            per_iteration[ncv] = info.seconds_cg / info.cg_iterations
    assert per_iteration[12] < per_iteration[24] * 4 / 3, per_iteration
