"""Eigenpairs of a degenerate spectrum over several thick restarts, from
several start vectors."""

import numpy as np
import pytest

import workloads as wl
from paper_1402_6297_gb300 import nfs as lib

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [1, 4, 5, 7, 9])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_degenerate_clusters_over_restarts(precision, seed):
    """omega = sqrt(Lambda_q) / 2, each twice, in a homogeneous medium at a
    k-point with degenerate clusters.  A_r V carried along by the recurrence
    over restarts drifts from A_r times V, and the re-orthogonalisation then
    works in a wrong inner product.  The tolerance: the values come from
    Rayleigh quotients, in error by the square of the vectors' error (1e-6 at
    most for the residual tolerances here)."""
    g = (16, 16, 16)
    n1, n2, n3 = g
    k = (0.5, 0.5, 5.0 / 12.0)
    tight = precision == "fp64"
    ctx = lib.Context(g, k, wl.homogeneous(g, eps=4.0), precision=precision, eig_tol=1e-12 if tight else 1e-10,
                      cg_tol=1e-13 if tight else 1e-12, deflation_checks=4, seed=seed)
    om, _, _ = ctx.eigs(8, vectors=False)
    ctx.close()
    i3, i2, i1 = np.meshgrid(np.arange(n3), np.arange(n2), np.arange(n1), indexing="ij")
    lq = sum(4 * np.sin(np.pi * (i + q) / n) ** 2 * n ** 2
             for i, q, n in ((i1, k[0], n1), (i2, k[1], n2), (i3, k[2], n3))).ravel()
    ref = np.sort(np.concatenate([np.sqrt(lq), np.sqrt(lq)]) / 2.0)[:8]
    assert np.abs(om - ref).max() < 1e-10 * ref.max(), (list(om), list(ref))
