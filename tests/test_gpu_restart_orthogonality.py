"""The vector that a thick restart goes on from."""

import numpy as np
import pytest

import workloads as wl
from oracle import gep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_it_is_orthogonalised_whatever_it_has_lost(lib, precision):
    """With a threshold that no loss of so short a basis reaches, one re-orthogonalisation is left per
    restart, of the last vector of the full basis; the eigenvalues are the
    oracle's (residuals of 1e-9 in the vectors, 1e-10 of the values at most)."""
    g = (8, 8, 8)
    k, med = (0.3, 0.2, 0.1), wl.chiral_sphere(g, 0.25, 13.0, 1.0, 0.5)
    with lib.Context(g, k, med, precision=precision, ncv=16, orth_tol=0.5, cg_tol=1e-12, eig_tol=1e-9) as c:
        omega, _, info = c.eigs(4, vectors=False)
    assert info.restarts >= 1
    assert info.reorthogonalisations >= info.restarts
    w, _, idx = gep.dense_eigs(g, k, med, 4)
    assert np.abs(omega - w[idx]).max() < 1e-10 * w[idx].max()
