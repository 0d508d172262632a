"""The adjoint kernel's integer sums against the oracle where their bookkeeping can go wrong: vector
counts around the carry (8) and the launch size (32), vectors whose sizes differ by many orders (the
running exponent), weights of either sign and zero, general lattices, and values that go to FP64.

Tolerance 1e-12 of the largest entry: a product rounds a few times at 2^-53, the oracle's strain some
30 times, and up to 40 vectors add up.
"""

import numpy as np
import pytest

from oracle import oracle as O
from workloads import complex_gaussian, fcc_lattice, two_phase_sphere

pytestmark = pytest.mark.gpu

KAPPA = (0.13, 0.27, 0.41)
IU = np.triu_indices(6)


def _run(N, block, xs, lam, w, a_lat=None):
    import torch
    import paper_2606_03599_gb300 as pc
    cell = two_phase_sphere(N, 0.35, 3)
    if a_lat is not None:
        cell.a_lat = a_lat
    h = pc.pc_grid_create(N, cell.C, cell.rho, phase=cell.phase, a_lat=cell.a_lat)
    try:
        C0, rho0, L = pc.pc_grid_units(h)
        pb = O.problem_from_cell(cell, C0=C0, rho0=rho0, L=L)
        pc.pc_set_k(h, KAPPA)
        n = N ** 3
        dC = torch.zeros(21 * n, dtype=torch.float64, device="cuda")
        dr = torch.zeros(n, dtype=torch.float64, device="cuda")
        pc.pc_eig_grad(h, block, torch.from_numpy(np.ascontiguousarray(xs)).reshape(-1).cuda(), lam, w, dC, dr)
        got = dC.view(21, n).T.cpu().numpy(), dr.cpu().numpy()
    finally:
        pc.pc_grid_destroy(h)
    ref = np.zeros((n, 21)), np.zeros(n)
    keep = np.zeros(n, bool)
    keep[np.arange(n) if block < 0 else O.block_index((N,) * 3, block)] = True
    with np.errstate(all="ignore"):
        for v in range(len(w)):
            X = xs[v] if block < 0 else O.inject(pb, block, xs[v])
            gC, gr = O.eigpair_gradients(pb, KAPPA, X, lam[v])
            ref[0][keep] += (w[v] * gC[:, IU[0], IU[1]] / (rho0 * L ** 2))[keep]
            ref[1][keep] += (w[v] * gr / rho0)[keep]
    return got, ref


@pytest.mark.parametrize("nvec", [1, 7, 8, 9, 31, 33, 40])
@pytest.mark.parametrize("block,lattice", [(-1, None), (2, "fcc")])
def test_vector_counts_and_sizes(nvec, block, lattice):
    N = 8
    m = N ** 3 if block < 0 else N ** 3 // 4
    rng = np.random.default_rng(nvec)
    xs = complex_gaussian((nvec, 3, m), nvec) * 10.0 ** rng.uniform(-12, 3, (nvec, 1, 1))
    w = rng.uniform(-2, 2, nvec)
    w[nvec // 2] = 0.0 if nvec > 1 else w[0]
    got, ref = _run(N, block, xs, rng.uniform(1e6, 1e8, nvec), w, fcc_lattice() if lattice else None)
    for a, b in zip(got, ref):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


@pytest.mark.parametrize("value", [1e-140, 1e140, 0.0, np.nan, np.inf])
def test_values_outside_the_integer_range(value):
    N, block = 8, 1
    xs = complex_gaussian((3, 3, N ** 3 // 4), 5)
    if np.isfinite(value):
        xs *= value
    else:
        xs[1, 2, 17] = value
    got, ref = _run(N, block, xs, np.array([1e7, 2e7, 3e7]), np.array([1.0, -0.5, 2.0]))
    for a, b in zip(got, ref):
        fine = np.isfinite(b)
        assert np.array_equal(fine, np.isfinite(a))
        assert np.abs(a[fine] - b[fine]).max() <= 1e-12 * np.abs(b[fine]).max()


def test_weights_outside_the_integer_range():
    N, block = 8, 0
    xs = complex_gaussian((2, 3, N ** 3 // 4), 6)
    got, ref = _run(N, block, xs, np.array([1e7, 2e7]), np.array([1e-200, 1e-201]))
    for a, b in zip(got, ref):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
