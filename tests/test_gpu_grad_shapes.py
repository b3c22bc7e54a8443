"""The gradient's sums over several vectors, on grids whose edges and z lengths
take different splits (the sums are kept in the order of the column kernel and
brought into natural order at the end), against the same quantities from the
eigenvector fields: with x = [E; H] of y, mu = 1 and omega' = 1 / (y^* B_r y),
d omega / d eps_c = -|E_c|^2 omega' and d omega / d gamma_c = 2 Im(conj(E_c) H_s(c))
omega', summed over the coupled pair in a pseudochiral medium.  The formulas hold
for any y; rounding of the two transforms and of sums of three leaves 1e-12 of
the largest entry."""

import numpy as np
import pytest

import workloads as wl

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kind", ["chiral", "xy", "xz", "yz"])
@pytest.mark.parametrize("n1,n3", [(8, 128), (12, 24), (16, 8), (24, 96), (32, 12), (48, 8), (64, 16), (96, 8), (128, 12)])
def test_against_the_fields(lib, n1, n3, kind):
    grid = (n1, n1, n3)
    pair = {"xy": (0, 1), "xz": (0, 2), "yz": (1, 2)}.get(kind)
    med = (wl.smoothed_chiral_field(grid, seed=3, sigma=0.12) if pair is None
           else wl.pseudochiral_cylinders(grid, 3, 0.2, 9.0, 1.5, 0.5, pair, 2))
    weights = np.array([0.7, -1.3, 0.4])
    gen = torch.Generator(device="cuda").manual_seed(n1 + n3)
    Y = torch.randn((3, 4 * n1 * n1 * n3), dtype=torch.complex128, device="cuda", generator=gen)
    with lib.Context(grid, (0.13, -0.21, 0.37), med) as c:
        d_eps, d_gamma = c.eig_grad(Y, weights)
        X = c.eig_fields(Y)
        s = torch.stack([torch.vdot(y, c.apply_Br(y)).real for y in Y])
    w = torch.from_numpy(weights).cuda() / s
    E, H = X[:, :3], X[:, 3:]
    shape = (-1, 1, 1, 1, 1)
    ref_eps = -(w.reshape(shape) * (E.abs() ** 2)).sum(0)
    swap = [0, 1, 2]
    if pair:
        swap[pair[0]], swap[pair[1]] = pair[1], pair[0]
    terms = (w.reshape(shape) * 2.0 * (E.conj() * H[:, swap]).imag).sum(0)
    ref_gamma = terms if pair is None else terms[pair[0]] + terms[pair[1]]
    for got, ref in ((d_eps, ref_eps), (d_gamma, ref_gamma)):
        assert torch.max(torch.abs(got.reshape(ref.shape) - ref)) < 1e-12 * torch.max(torch.abs(ref))
