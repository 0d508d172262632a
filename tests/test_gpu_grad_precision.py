"""The adjoint kernel's 21 sums at every node against extended precision, each entry against its own size: small
strains, small parts and small vectors next to large ones keep the digits that FP64 gives them.

Tolerance, entry (p, r) of a node: the strain of component values X whose differences are G takes 8 roundings of
2^-53 G and one of 2^-53 X where a Bloch phase or an alignment touches the values (a third of the cases have none
of the first kind); products, weights and up to 12 additions another 20 of 2^-53 |e_p| |e_r|.
"""

import numpy as np
import pytest

from oracle import oracle as O
from workloads import complex_gaussian, fcc_lattice, two_phase_sphere

pytestmark = pytest.mark.gpu

LD, CLD = np.longdouble, np.clongdouble
IU = list(zip(*np.triu_indices(6)))
SIGNS = [(1, 1), (1, -1), (-1, 1), (-1, -1)]
CSL = [(1, 1, 1, 1), (1, 1, -1, -1), (1, -1, 1, -1)]


def moved(x, d, phi):
    for axis, step, ph in ((-1, d[0], phi[0]), (-2, d[1], phi[1]), (-3, d[2], phi[2])):
        x = np.roll(x, -step, axis=axis)
        at = [slice(None)] * x.ndim
        at[axis] = x.shape[axis] - 1 if step > 0 else 0
        x[tuple(at)] *= CLD(complex(np.cos(ph), step * np.sin(ph)))
    return x


def strain(x, N, phi, mix):
    """Six strains of x [3, N^3] and a bound on the roundings of each (per node, before 2^-53)."""
    x = x.reshape(3, N, N, N).astype(CLD)
    H, S, X = [0, 0, 0], 0, np.abs(x)
    for l, (s2, s3) in enumerate(SIGNS):
        n = moved(x, (-1, -s2, -s3), phi)
        g = n - x
        S, X = S + np.abs(g), np.maximum(X, np.abs(n))
        for s in range(3):
            H[s] = H[s] + CSL[s][l] * g
    G = [sum(LD(mix[s][m]) * H[s] for s in range(3)) for m in range(3)]
    B = [sum(abs(mix[s][m]) for s in range(3)) * (8 * S + X) for m in range(3)]
    pick = lambda Q: [Q[0][0], Q[1][1], Q[2][2], Q[2][1] + Q[1][2], Q[2][0] + Q[0][2], Q[1][0] + Q[0][1]]
    return [e.reshape(-1) for e in pick(G)], [b.reshape(-1) for b in pick(B)]


@pytest.mark.parametrize("what", ["component", "imag", "vectors", "planes", "uniform", "weights"])
@pytest.mark.parametrize("block,lattice", [(-1, "cubic"), (2, "fcc"), (1, "cubic")])
@pytest.mark.parametrize("small", [1e-6, 1e-11])
def test_every_entry_on_its_own_scale(what, block, lattice, small):
    import torch
    import paper_2606_03599_gb300 as pc
    N, nvec = 8, 12
    n = N ** 3
    cell = two_phase_sphere(N, 0.35, 3)
    if lattice == "fcc":
        cell.a_lat = fcc_lattice()
    rng = np.random.default_rng(int(-np.log10(small)))
    idx = np.arange(n) if block < 0 else O.block_index((N,) * 3, block)
    kappa = (0.0, 0.0, 0.0) if what in ("imag", "uniform") else (0.13, 0.27, 0.41)
    xs = np.zeros((nvec, 3, n), complex)
    xs[:, :, idx] = complex_gaussian((nvec, 3, len(idx)), 5)
    w = rng.uniform(-2, 2, nvec)
    if what == "component":
        xs[:, 2] *= small
    elif what == "imag":
        xs = xs.real + 1j * small * xs.imag
    elif what == "vectors":
        xs *= small ** rng.uniform(0, 1, (nvec, 1, 1))
    elif what == "planes":
        xs *= small ** (np.arange(n) // (N * N) / N)
    elif what == "uniform":
        xs[:, 0] = 0
        xs[:, 0][:, idx] = 1.0
        xs[:, 1:] *= small
    else:
        w *= small ** rng.uniform(0, 1, nvec)
    h = pc.pc_grid_create(N, cell.C, cell.rho, phase=cell.phase, a_lat=cell.a_lat)
    try:
        C0, rho0, L = pc.pc_grid_units(h)
        pc.pc_set_k(h, kappa)
        dC = torch.zeros(21 * n, dtype=torch.float64, device="cuda")
        dr = torch.zeros(n, dtype=torch.float64, device="cuda")
        x = torch.from_numpy(np.ascontiguousarray(xs[:, :, idx])).reshape(-1).cuda()
        pc.pc_eig_grad(h, block, x, rng.uniform(1e6, 1e8, nvec), w, dC, dr)
        got = dC.view(21, n).cpu().numpy()
    finally:
        pc.pc_grid_destroy(h)
    ainv = np.linalg.inv(cell.a_lat / L)
    mix = [[ainv[s, m] * N / 4 for m in range(3)] for s in range(3)]
    phi = [2 * np.pi * (k - np.floor(k)) for k in kappa]
    ref, tol = np.zeros((21, n), LD), np.zeros((21, n), LD)
    for v in range(nvec):
        e, b = strain(xs[v], N, phi, mix)
        f = LD(w[v]) / (LD(rho0) * LD(L) * LD(L))
        for q, (p, r) in enumerate(IU):
            two = 1 if p == r else 2
            ref[q] += two * f * (np.conj(e[p]) * e[r]).real
            # parts apart: an imaginary strain's product does not excuse a real one's error
            ep, er = np.abs(e[p]), np.abs(e[r])
            tol[q] += two * abs(f) * (b[p] * er + ep * b[r] + 20 * ep * er)
    assert (np.abs(got[:, idx] - ref[:, idx]) <= 2.0 ** -53 * tol[:, idx]).all()
    outside = np.setdiff1d(np.arange(n), idx)
    assert not got[:, outside].any()
