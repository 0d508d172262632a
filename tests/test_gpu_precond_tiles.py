"""The complex128 preconditioner's pencil tiles: one block alone and the four blocks together take different tiles
(by the number of CTAs and the divisors of N / 2) and give the same values, which are the oracle's.

A value's arithmetic does not depend on its tile, so alone = together exactly; 1e-12 of the norm against the oracle,
as in test_gpu_precond.py.
"""

import numpy as np
import pytest

from oracle import oracle as O
from workloads import complex_gaussian, two_phase_sphere

pytestmark = pytest.mark.gpu

KAPPA = (0.21, 0.33, 0.14)


# N / 2: 5, 13, 25 no divisor from two to four; 12 compiled factors; 18 small tiles in both; 36 and 39 large tiles for
# four systems only
@pytest.mark.parametrize("N", [10, 24, 26, 36, 50, 72, 78])
def test_one_block_equals_the_block_among_four(N):
    import torch
    import paper_2606_03599_gb300 as pc
    cell = two_phase_sphere(N, 0.35, 3)
    h = pc.pc_grid_create(N, cell.C, cell.rho, phase=cell.phase, a_lat=cell.a_lat)
    try:
        pc.pc_set_k(h, KAPPA)
        x = complex_gaussian((3, N ** 3), 5)
        full = torch.from_numpy(x).reshape(-1).cuda()
        out = torch.zeros_like(full)
        pc.pc_block_precond(h, -1, -0.5, full, out)
        got = out.cpu().numpy().reshape(3, -1)
        for b in range(4):
            idx = O.block_index((N,) * 3, b)
            xb = torch.from_numpy(np.ascontiguousarray(x[:, idx])).reshape(-1).cuda()
            yb = torch.zeros_like(xb)
            pc.pc_block_precond(h, b, -0.5, xb, yb)
            one = yb.cpu().numpy().reshape(3, -1)
            assert np.array_equal(one, got[:, idx])
        if N <= 26:
            C0, rho0, L = pc.pc_grid_units(h)
            pb = O.problem_from_cell(cell, C0=C0, rho0=rho0, L=L)
            ref = O.precond_full(pb, KAPPA, -0.5, x).reshape(3, -1)
            assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
    finally:
        pc.pc_grid_destroy(h)
