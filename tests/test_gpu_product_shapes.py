"""The A_r product over grids, media and element types at the edges of its
tiles: every plane edge with the shortest, an odd and the longest z lengths
(one- and two-stage line DFTs, one and two x slots per column CTA), each
pseudochiral axis pair, mu present and absent, against the CPU oracle.
Tolerances as in test_gpu_matvec: relative to the largest entry, 1e-12
(complex128 and double-single), 2e-5 (complex64).  The solve checks the CG form
of the same kernels by its true residual."""

import numpy as np
import pytest

import workloads as wl
from oracle import nfgep

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

K = (0.13, -0.21, 0.37)
SHAPES = [(8, 128), (12, 8), (16, 96), (24, 24), (24, 64), (32, 12), (48, 16), (64, 8), (96, 8), (96, 24), (128, 8)]
MEDIA = ["chiral", "xy", "xz", "yz"]


def medium(kind, grid, mu):
    m = (wl.smoothed_chiral_field(grid, seed=3, sigma=0.12) if kind == "chiral"
         else wl.pseudochiral_cylinders(grid, 3, 0.2, 9.0, 1.5, 0.5, {"xy": (0, 1), "xz": (0, 2), "yz": (1, 2)}[kind], 2))
    if mu:
        m = wl.Medium(m.grid, m.kind, m.eps, m.gamma, 1.0 + 0.5 * np.random.default_rng(4).random(m.eps.shape), m.axes)
    return m


def rel(a, b):
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("i", range(len(SHAPES)), ids=["%dx%d" % s for s in SHAPES])
def test_product(lib, i):
    n1, n3 = SHAPES[i]
    grid = (n1, n1, n3)
    med = medium(MEDIA[i % 4], grid, mu=i % 3 == 0)
    orc = nfgep.NFGEP(grid, K, med)
    ctx = lib.Context(grid, K, med, precision="mixed", cg_tol=1e-11)
    u = wl.random_complex(4 * ctx.n, 7)
    ref = orc.Ar(u)
    ud = torch.from_numpy(u).cuda()
    assert rel(ctx.matvec(ud).cpu().numpy(), ref) < 1e-12
    assert rel(ctx.matvec_ds(ud).cpu().numpy(), ref) < 1e-12
    assert rel(ctx.matvec(ud.to(torch.complex64)).cpu().numpy(), ref) < 2e-5
    if n1 * n1 * n3 <= 20000:
        x, info = ctx.cg_solve(ud)
        assert info.status == 0
        assert np.linalg.norm(orc.Ar(x.cpu().numpy()) - u) < 1.1e-11 * np.linalg.norm(u)
    ctx.close()


@pytest.mark.parametrize("kind", MEDIA)
def test_solves_of_a_batch_match_single_problems(lib, kind):
    """A batch of three problems through the same launches gives each problem's
    own eigenvalues (per-problem strides of the workspace, material and CG state)."""
    grid = (16, 16, 24)
    ks = [K, (0.3, 0.2, 0.1), (0.45, 0.05, 0.25)]
    media = [medium(kind, grid, mu=True) for _ in ks]
    for j, m in enumerate(media):
        m.eps[...] = m.eps * (1.0 + 0.1 * j)
    b = lib.Batch(list(zip([grid] * 3, ks, media)), precision="mixed")
    om, _ = b.eigs(3)
    b.close()
    for j in range(3):
        ctx = lib.Context(grid, ks[j], media[j], precision="mixed")
        one = ctx.eigs(3, vectors=False)[0]
        ctx.close()
        assert np.abs(om[j] - one).max() < 1e-10 * one.max()
