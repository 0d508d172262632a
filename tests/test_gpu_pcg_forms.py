"""The PCG iteration's forms give the same eigenvalues: step lengths summed in the vector kernels (small
solves) or by kernels of their own (large ones), with the complex64 preconditioner (flexible beta) and
the FP64 one, over fused, own and library transforms, blocks and full space.

Tolerance 2e-8: every solve's true relative residual is at most 1e-8, and an eigenvalue is off by no
more than its residual.
"""

import numpy as np
import pytest

from workloads import two_phase_sphere

pytestmark = pytest.mark.gpu

KAPPAS = np.array([[0.5, 0.0, 0.0], [0.3, 0.1, 0.2], [0.2, 0.45, 0.1]])


# N / 2 = 4 and 12: fused; 11: own transform, not fused; 17: library transform; 20: fused, more than
# two CTAs per SM with three Bloch vectors
@pytest.mark.parametrize("N,nk", [(8, 1), (24, 1), (22, 1), (34, 1), (40, 3)])
@pytest.mark.parametrize("full", [0, 1])
def test_forms_agree(N, nk, full):
    import paper_2606_03599_gb300 as pc
    if full and N > 24:
        pytest.skip("the full space at the small sizes")
    cell = two_phase_sphere(N, 0.35, 2)
    h = pc.pc_grid_create(N, cell.C, cell.rho, phase=cell.phase, a_lat=cell.a_lat)
    try:
        got = []
        for fp32 in (1, 0):
            opt = pc.pc_options_default(precond_fp32=fp32, full_space=full)
            if nk == 1:
                ev, _, info = pc.pc_eigs(h, KAPPAS[1], 8, opt=opt)
            else:
                ev, _, _ = pc.pc_eigs_multi(h, KAPPAS[:nk], 8, opt=opt)
            got.append(np.asarray(ev))
        assert np.abs(got[0] - got[1]).max() <= 2e-8 * np.abs(got[1]).max()
    finally:
        pc.pc_grid_destroy(h)
