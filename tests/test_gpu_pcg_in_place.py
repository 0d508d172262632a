"""The PCG iteration with its step lengths summed inside the vector kernels (few CTAs) and by kernels of their own
(many) runs the same recurrence: iterates, counts and exits against a plain loop over the public operator and
preconditioner, on both sides of the line (304 vector CTAs of 1024 values on a GPU of 152 SMs), and the same band solve alone
(in place) and among sixteen Bloch vectors (kernels of their own).

Tolerances.  Two runs of the same recurrence in FP64 differ by its rounding, which grows with the residual's fall; after
7 iterations (a fall of about 1e3) the iterates agree to 1e-12 of their norm with two digits to spare.  Eigenvalues whose
residual is at most 1e-8 agree to its square times the spectrum's spread, 1e-12; 1e-10 is asked for.
"""

import numpy as np
import pytest

from workloads import two_phase_sphere

pytestmark = pytest.mark.gpu

KAPPA = (0.3, 0.2, 0.1)
PC_OK, PC_ENOCONV, PC_EBREAKDOWN = 0, -4, -5


def grid(pc, N):
    cell = two_phase_sphere(N, 0.35, 2)
    h = pc.pc_grid_create(N, cell.C, cell.rho, phase=cell.phase, a_lat=cell.a_lat)
    pc.pc_set_k(h, KAPPA)
    return h


def plain_pcg(pc, h, block, sigma, b, maxit):
    """x, iterations and whether p^H (A - sigma M) p <= 0 or Re<r, z> <= 0 ended it."""
    import torch
    dot = lambda u, v: float(torch.vdot(u, v).real)
    x, r = torch.zeros_like(b), b.clone()
    z, q = torch.empty_like(b), torch.empty_like(b)
    pc.pc_block_precond(h, block, sigma, r, z)
    p, rz = z.clone(), dot(r, z)
    for it in range(maxit):
        pc.pc_block_apply(h, block, p, q, shift=sigma)
        pq = dot(p, q)
        if not pq > 0:
            return x, it, True
        x += (rz / pq) * p
        r -= (rz / pq) * q
        pc.pc_block_precond(h, block, sigma, r, z)
        new = dot(r, z)
        if not new > 0:
            return x, it + 1, True
        p = z + (new / rz) * p
        rz = new
    return x, maxit, False


# 12, 96, 286 vector CTAs: in place; 354 and 648: kernels of their own
@pytest.mark.parametrize("N", [16, 44, 72, 78, 96])
@pytest.mark.parametrize("maxit", [1, 2, 3, 4, 7])
def test_iterates_at_the_iteration_limit(N, maxit):
    import torch
    import paper_2606_03599_gb300 as pc
    h = grid(pc, N)
    try:
        gen = torch.Generator(device="cuda").manual_seed(N)
        b = torch.randn(3 * N ** 3 // 4, dtype=torch.complex128, device="cuda", generator=gen)
        sigma = pc.pc_default_sigma(h)
        x = torch.zeros_like(b)
        info = pc.pc_shift_invert_pcg(h, 1, sigma, b, x, tol=1e-14, maxit=maxit, raise_on_fail=False)
        ref, its, broke = plain_pcg(pc, h, 1, sigma, b, maxit)
        assert not broke and info["rc"] == PC_ENOCONV and info["iters"] == its == maxit
        assert float((x - ref).norm()) <= 1e-12 * float(ref.norm())
        res = torch.empty_like(b)
        pc.pc_block_apply(h, 1, x, res, shift=sigma)
        true = float((b - res).norm() / b.norm())
        assert abs(info["rel_resid"] - true) <= 1e-10
    finally:
        pc.pc_grid_destroy(h)


@pytest.mark.parametrize("N", [16, 44, 78])
def test_breakdown_keeps_the_last_iterate(N):
    """A shift above the lowest eigenvalue and below the reference medium's: the operator is indefinite and the
    preconditioner is not, so the solve meets p^H (A - sigma M) p <= 0 after some steps."""
    import torch
    import paper_2606_03599_gb300 as pc
    h = grid(pc, N)
    try:
        C0, rho0, L = pc.pc_grid_units(h)
        ev, block_of, _ = pc.pc_eigs(h, KAPPA, 4)
        block = int(block_of[0])
        sigma = 1.03 * float(ev[0]) * rho0 * L * L / C0
        pc.pc_set_k(h, KAPPA)
        gen = torch.Generator(device="cuda").manual_seed(3)
        b = torch.randn(3 * N ** 3 // 4, dtype=torch.complex128, device="cuda", generator=gen)
        ref, its, broke = plain_pcg(pc, h, block, sigma, b, 200)
        assert broke and its > 1
        x = torch.zeros_like(b)
        info = pc.pc_shift_invert_pcg(h, block, sigma, b, x, tol=1e-14, maxit=200, raise_on_fail=False)
        assert info["rc"] == PC_EBREAKDOWN and abs(info["iters"] - its) <= 1
        # the same iterate, stopped before the step that would have gone up: finite and as large
        assert bool(torch.isfinite(torch.view_as_real(x)).all())
        assert float((x - ref).norm()) <= 1e-6 * float(ref.norm())
    finally:
        pc.pc_grid_destroy(h)


@pytest.mark.parametrize("fp32", [0, 1])
@pytest.mark.parametrize("N", [12, 16])
def test_a_solve_alone_equals_the_same_solve_among_sixteen(N, fp32):
    """Systems that finish at different iterations in one launch, in both forms."""
    import paper_2606_03599_gb300 as pc
    h = grid(pc, N)
    try:
        opt = pc.pc_options_default(precond_fp32=fp32)
        kappas = np.random.default_rng(1).uniform(0.05, 0.45, (16, 3))
        many, _, infos = pc.pc_eigs_multi(h, kappas, 8, opt=opt)
        solves = iters = 0
        for i in range(16):
            ev, _, info = pc.pc_eigs(h, kappas[i], 8, opt=opt)
            assert np.abs(ev - many[i]).max() <= 1e-10 * np.abs(ev).max()
            solves, iters = solves + info["inner_solves"], iters + info["pcg_iters"]
        # the counts of a solve in lockstep are those of all its vectors: the iterations per solve agree
        assert abs(iters / solves - infos[0]["pcg_iters"] / infos[0]["inner_solves"]) <= 0.02 * iters / solves
    finally:
        pc.pc_grid_destroy(h)
