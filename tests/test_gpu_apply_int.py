"""The integer-pipe complex128 apply's two launch forms on the GPU: a vector alone (two threads per
cell) and the same vector in a batch that fills the GPU (one thread per cell) give the same result, and
both the oracle's.

Tolerance: a node's integer arithmetic is the same in both forms, so alone = batched exactly; the
oracle's FP64 chain is some 60 roundings of 2^-53, both sides 1.4e-14 of the output's norm.  A node
out of the integers' range sends its column's next planes to FP64 up to the end of its CTA's planes,
which the two forms cut differently: there each is within 4 x 1.4e-14 of the oracle's largest value,
the bound that the CPU test of such nodes has.
"""

import numpy as np
import pytest

from oracle import oracle as O
from workloads import complex_gaussian, fcc_lattice, two_phase_sphere

pytestmark = pytest.mark.gpu

KAPPA = (0.21, -0.33, 0.4)


@pytest.mark.parametrize("N,count", [(4, 330), (8, 170), (18, 70), (34, 40)])
@pytest.mark.parametrize("lattice", ["cubic", "fcc"])
@pytest.mark.parametrize("special", [None, 1e-300, 1e300])
def test_one_vector_equals_the_same_vector_in_a_batch(N, count, lattice, special):
    import torch
    import paper_2606_03599_gb300 as pc
    cell = two_phase_sphere(N, 0.35, 3)
    if lattice == "fcc":
        cell.a_lat = fcc_lattice()
    block = 1
    idx = O.block_index((N,) * 3, block)
    x = complex_gaussian((3, N ** 3), 5)[:, idx]
    if special is not None:
        x[:, len(idx) // 2] *= special  # one node out of the integer range
    h = pc.pc_grid_create(N, cell.C, cell.rho, phase=cell.phase, a_lat=cell.a_lat)
    try:
        C0, rho0, L = pc.pc_grid_units(h)
        pb = O.problem_from_cell(cell, C0=C0, rho0=rho0, L=L)
        pc.pc_set_k(h, KAPPA)
        d = torch.from_numpy(np.ascontiguousarray(x)).reshape(-1).cuda()
        many = d.repeat(count)
        ys, alone = torch.zeros_like(many), torch.zeros_like(d)
        pc.pc_block_apply(h, block, d, alone, shift=0.7)
        pc.pc_block_apply_many(h, block, count, many, ys, shift=0.7)
        torch.cuda.synchronize()
        got = alone.cpu().numpy().reshape(3, -1)
        first, last = (ys.view(count, 3, -1)[i].cpu().numpy() for i in (0, -1))
        same = bool((ys.view(count, -1) == alone).all())
    finally:
        pc.pc_grid_destroy(h)
    ref = O.apply_block(pb, KAPPA, block, x, 0.7)
    if special is None:
        assert same
        assert np.linalg.norm(got - ref) <= 1.4e-14 * np.linalg.norm(ref)
    else:
        for y in (got, first, last):
            assert np.abs(y - ref).max() <= 4 * 1.4e-14 * np.abs(ref).max()
