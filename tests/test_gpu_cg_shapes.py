"""The CG form of the product's kernels at every plane edge: the tiles, and the
partial sums, whose number goes up to the room for them (3072 of p^* A_r p at
edge 128, 2048 of r^* r at 128^3 in complex128).  The residual of a solve by the
complex128 product (whose parity with the oracle test_gpu_product_shapes checks)
is within the tolerance, and a tenth of it for rounding, as there."""

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

K = (0.13, -0.21, 0.37)
SHAPES = [(8, 12), (12, 128), (16, 8), (24, 12), (32, 8), (32, 96), (48, 8), (48, 96), (64, 8), (96, 8), (128, 8), (128, 128)]


def medium(i, grid):
    if i % 3 == 0:
        return wl.pseudochiral_cylinders(grid, 3, 0.2, 9.0, 1.5, 0.5, ((0, 1), (0, 2), (1, 2))[i // 3 % 3], 2)
    m = wl.chiral_sphere(grid, 0.25, 13.0, 1.0, 0.5)
    if i % 3 == 1:
        m = wl.Medium(m.grid, m.kind, m.eps, m.gamma, 1.0 + 0.5 * np.random.default_rng(4).random(m.eps.shape), m.axes)
    return m


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("i", range(len(SHAPES)), ids=["%dx%d" % s for s in SHAPES])
def test_solve(lib, i, precision):
    n1, n3 = SHAPES[i]
    grid = (n1, n1, n3)
    with lib.Context(grid, K, medium(i, grid), precision=precision, cg_tol=1e-11) as c:
        gen = torch.Generator(device="cuda").manual_seed(i)
        b = torch.randn(4 * n1 * n1 * n3, dtype=torch.complex128, device="cuda", generator=gen)
        x, info = c.cg_solve(b)
        assert info.status == lib.NFS_OK and info.iterations > 8
        assert torch.linalg.norm(c.matvec(x) - b) < 1.1e-11 * torch.linalg.norm(b)


@pytest.mark.parametrize("precision,grid,problems", [
    ("fp64", (8, 8, 8), 2), ("fp64", (8, 8, 8), 3),          # kernels that overlap, and one problem more
    ("fp64", (12, 12, 12), 1), ("fp64", (12, 12, 12), 2),    # likewise
    ("fp64", (128, 128, 8), 2), ("mixed", (128, 128, 8), 2)])
def test_batches_match_single_problems(lib, precision, grid, problems):
    ks = [K, (0.3, 0.2, 0.1), (0.45, 0.05, 0.25)][:problems]
    media = [medium(1, grid) for _ in ks]
    for j, m in enumerate(media):
        m.eps[...] = m.eps * (1.0 + 0.1 * j)
    with lib.Batch(list(zip([grid] * problems, ks, media)), precision=precision) as b:
        om, _ = b.eigs(2)
    for j in range(problems):
        with lib.Context(grid, ks[j], media[j], precision=precision) as c:
            one = c.eigs(2, vectors=False)[0]
        assert np.abs(om[j] - one).max() < 1e-10 * one.max()
