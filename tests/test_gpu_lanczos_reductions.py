"""The reductions of an eigensolve (exact inner products with the basis, the
start of the inner solves, Rayleigh-Ritz over all problems of a batch) at basis
sizes and batch sizes around their tiles."""

import numpy as np
import pytest

import workloads as wl
from oracle import gep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("problems", [1, 3])
@pytest.mark.parametrize("ncv", [9, 17, 40])
def test_every_step_orthogonalised(lib, precision, problems, ncv):
    """orth_tol = 0 removes what the exact inner products find in every step:
    a wrong or missing one (odd counts, the last vector, the change of the
    block count at 16 vectors) ruins the basis within a few steps.  Tolerance:
    residuals of 1e-8 in the vectors give eigenvalues to their square."""
    g = (8, 8, 8)
    ks = wl.bz_path_midpoints(problems)
    probs = [(g, tuple(k), wl.chiral_sphere(g, 0.25, 13.0, 1.0, 0.3 + 0.1 * i)) for i, k in enumerate(ks)]
    with lib.Batch(probs, precision=precision, ncv=ncv, orth_tol=0.0, cg_tol=1e-11, eig_tol=1e-8) as b:
        omega, infos = b.eigs(4)
    for i, (_, k, med) in enumerate(probs):
        w, _, idx = gep.dense_eigs(g, k, med, 4)
        assert np.abs(omega[i] - w[idx]).max() / w[idx].min() < 1e-9, (i, list(omega[i]), list(w[idx]))
        assert infos[i].reorthogonalisations > 0
