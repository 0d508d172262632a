"""The work that a user of the band solver has it do, as cases that can be timed.

Each case goes through the package's entry points as a program calls them: the block operator on
one vector and on batches, the reference-medium preconditioner, one shift-invert solve, whole band
solves at several sizes and precisions, and the eigenvalue-gradient (adjoint) call.  Grid sizes are
those of the repository's own workloads (N = 8, 48, 60, 64, 96, 128, 160); ``draw`` spreads them
over the even sizes between, ragged ones among them.

``exact`` evaluates the same quantities in complex128 with plain torch on the full grid, written
from the operator's definition: body-diagonal Bloch differences, strain, nodewise stiffness,
adjoint differences.
"""

import math

import numpy as np
import torch

import paper_2606_03599_gb300 as pc

GPA = 1.0e9
C0, RHO0 = 1.0e9, 1.0e3  # hat units: stiffness / 1 GPa, density / 1000 kg/m^3, lengths / |det A|^(1/3)
NEV_DENSE_N = 16         # largest grid whose dense spectrum exact() computes


def listed():
    return [
        # One operator application on a coarse grid: the smallest call a program makes.
        {"name": "apply_c128_n8_one", "kind": "apply", "N": 8, "dtype": "c128", "material": "phase", "block": 1, "count": 1},
        # One vector per parity block at the fine-grid size of the precision workload, complex64.
        {"name": "apply_c64_n160_blocks", "kind": "apply", "N": 160, "dtype": "c64", "material": "phase", "block": 4, "count": 4},
        # The operator launch of a lockstep band solve: many vectors of a 48^3 grid, FP64.
        {"name": "apply_c128_n48_many", "kind": "apply", "N": 48, "dtype": "c128", "material": "phase", "block": 2, "count": 64},
        # The same in complex64 (the inner solves of the mixed-precision mode).
        {"name": "apply_c64_n48_many", "kind": "apply", "N": 48, "dtype": "c64", "material": "phase", "block": 1, "count": 64},
        # Sub-pixel fractions on an FCC lattice, ragged quarter grid (30 wide), FP64.
        {"name": "apply_c128_fcc_n60", "kind": "apply", "N": 60, "dtype": "c128", "material": "fcc", "block": 4, "count": 4},
        # Every node its own stiffness (the differentiation workload's grid), full space, FP64.
        {"name": "apply_c128_nodewise_n64", "kind": "apply", "N": 64, "dtype": "c128", "material": "nodewise", "block": -1, "count": 1},
        # The preconditioner of the inner solves at the largest size of the batching workload.
        {"name": "precond_c64_n128", "kind": "precond", "N": 128, "dtype": "c64", "fp32": False, "block": 0},
        # One FP64 shift-invert solve.
        {"name": "pcg_c128_n48", "kind": "pcg", "N": 48, "block": 3},
        # A whole band solve of the smallest workload: one Bloch vector, 12 bands, FP64.
        {"name": "bands_fp64_n8", "kind": "bands", "N": 8, "nk": 1, "nev": 12, "precision": "fp64"},
        # The headline: Bloch vectors of the simple-cubic path in lockstep, 20 bands, FP64.
        {"name": "bands_fp64_n48", "kind": "bands", "N": 48, "nk": 4, "nev": 20, "precision": "fp64"},
        # A fine grid in mixed precision, 16 bands (batching workload's largest grid).
        {"name": "bands_mixed_n128", "kind": "bands", "N": 128, "nk": 1, "nev": 16, "precision": "mixed"},
        # The backward pass of the differentiation workload: 12 eigenvectors on 64^3 nodes.
        {"name": "grad_n64", "kind": "grad", "N": 64, "material": "phase", "block": -1, "count": 12},
    ]


def _even(rng, lo, hi):
    """An even size between lo and hi, spread over its logarithm."""
    return max(lo, min(hi, 2 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "apply", "precond", "pcg", "bands", "bands", "grad"])
    if kind == "apply":
        material = rng.choice(["phase", "phase", "fcc", "nodewise"])
        dtype = "c128" if material == "nodewise" else rng.choice(["c64", "c128"])
        block = rng.choice([-1, 0, 1, 2, 3, 4])
        N = _even(rng, 8, 160 if block >= 0 else 96)
        per = N ** 3 if block == -1 else N ** 3 // 4
        most = max(1, min(64, 4 * 10 ** 6 // per))
        count = 4 if block == 4 else max(1, min(most, round(math.exp(rng.uniform(0, math.log(most + 0.5))))))
        return {"kind": kind, "N": N, "dtype": dtype, "material": material, "block": block, "count": count}
    if kind == "precond":
        dtype = rng.choice(["c64", "c128"])
        return {"kind": kind, "N": _even(rng, 8, 128), "dtype": dtype, "fp32": dtype == "c128" and rng.random() < 0.5,
                "block": rng.choice([-1, 0, 1, 2, 3])}
    if kind == "pcg":
        return {"kind": kind, "N": _even(rng, 8, 64), "block": rng.choice([0, 1, 2, 3])}
    if kind == "grad":
        N = _even(rng, 8, 64)
        return {"kind": kind, "N": N, "material": rng.choice(["phase", "fcc"]), "block": rng.choice([-1, 0, 1, 2, 3]),
                "count": rng.randint(1, 12)}
    N = _even(rng, 8, 48)
    # several Bloch vectors together where the grid's transform length N/2 has small factors only
    nk = rng.randint(1, 4) if N // 2 in (4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16, 18, 20, 21, 22, 24) else 1
    return {"kind": kind, "N": N, "nk": nk, "nev": rng.choice([8, 12, 16, 20]) if N > 10 else 12,
            "precision": rng.choice(["fp64", "mixed"])}


# ---------------------------------------------------------------------------------- inputs
def _kappas(seed, nk):
    """Bloch vectors inside the zone (reduced coordinates), away from its centre."""
    rng = np.random.default_rng(seed + 77)
    return rng.uniform(0.12, 0.48, size=(nk, 3))


def _material(case, seed):
    """Two-phase cell: an anisotropic sphere in an isotropic matrix, as phase ids, as sub-pixel
    fractions on an FCC lattice, or written out node by node."""
    N, kind = case["N"], case.get("material", "phase")
    rng = np.random.default_rng(seed)
    Q, R = np.linalg.qr(rng.standard_normal((6, 6)))
    Q = Q * np.sign(np.diag(R))[None, :]
    C1 = (Q * (rng.uniform(20, 200, 6) * GPA)[None, :]) @ Q.T
    C = np.zeros((2, 6, 6))
    C[0, :3, :3] = 40 * GPA
    C[0, range(6), range(6)] = [100 * GPA] * 3 + [30 * GPA] * 3
    C[1] = 0.5 * (C1 + C1.T)
    rho = np.array([1200.0, 7800.0])
    A = np.eye(3)
    if kind == "fcc":
        A = 0.015 * (np.ones((3, 3)) - np.eye(3))
    g = (np.arange(N) - N // 2) / N
    r = np.stack(np.meshgrid(g, g, g, indexing="ij")[::-1], axis=-1).reshape(-1, 3)  # i fastest
    a0 = np.abs(np.linalg.det(A)) ** (1 / 3)
    d = np.linalg.norm(r @ A.T, axis=1) / a0
    if kind == "phase":
        return A, C, rho, (d <= 0.35 * (1 + 1e-12)).astype(np.uint8)
    return A, C, rho, np.clip((0.35 - d) * N + 0.5, 0.0, 1.0).astype(np.float32)


IU = np.triu_indices(6)


def _nodewise(C, rho, theta):
    """(N^3, 21) stiffness and (N^3,) density of the two-phase mixture with theta in 64 bits."""
    th = theta.astype(np.float64)
    return (1 - th)[:, None] * C[0][IU] + th[:, None] * C[1][IU], (1 - th) * rho[0] + th * rho[1]


def _blocks(case):
    return [0, 1, 2, 3] if case["block"] == 4 else [case["block"]]


def _vectors(case, seed, kappa, blocks, per_block):
    """Vectors as a Krylov solve meets them: a few long Bloch waves and broad-band noise.  One
    tensor [per_block][3][m] for each entry of `blocks`."""
    N = case["N"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    pos = torch.arange(N, device="cuda", dtype=torch.float64) / N
    for b in blocks:
        m = N ** 3 if b < 0 else N ** 3 // 4
        idx = None if b < 0 else _block_nodes(N, b)
        x = torch.empty(per_block, 3, m, dtype=torch.complex128, device="cuda")
        for v in range(per_block):
            noise = torch.randn(2, 3, m, generator=gen, device="cuda", dtype=torch.float64)
            x[v] = 0.1 * torch.complex(noise[0], noise[1])
            amp = torch.randn(2, 3, 3, generator=gen, device="cuda", dtype=torch.float64)
            for w in range(3):
                q = [kappa[l] + (1 if l == w else 0) for l in range(3)]
                e = [torch.exp(2j * math.pi * q[l] * pos) for l in range(3)]
                wave = (e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]).reshape(-1)
                wave = wave if idx is None else wave[idx]
                x[v] += torch.complex(amp[0, w], amp[1, w])[:, None] * wave[None, :]
        out.append(x.to(torch.complex64) if case.get("dtype") == "c64" else x)
    return out


def _block_nodes(N, b):
    i = torch.arange(N, device="cuda")
    k, j, i = torch.meshgrid(i, i, i, indexing="ij")
    return torch.nonzero((((i + j) % 2 == b >> 1) & ((i + k) % 2 == b & 1)).reshape(-1)).reshape(-1)


def _hat(A):
    L = abs(np.linalg.det(A)) ** (1 / 3)
    return L, np.linalg.inv(A / L)


def _shift(C, rho):
    """The default shift: -0.30 max |C| / max rho in hat units."""
    return -0.30 * (np.abs(C).max() / C0) / (rho.max() / RHO0)


class Grid:
    """A grid handle that is given back with its state."""

    def __init__(self, case, A, C, rho, th):
        kind = case.get("material", "phase")
        if kind == "nodewise":
            c21, rn = _nodewise(C, rho, th)
            self.h = pc.pc_grid_create_nodewise(case["N"], c21, rn, a_lat=A)
        else:
            self.h = pc.pc_grid_create(case["N"], C, rho, a_lat=A, **({"phase": th} if kind == "phase" else {"theta": th}))

    def __del__(self):
        if getattr(self, "h", None):
            pc.pc_grid_destroy(self.h)
            self.h = None


def prepare(case, seed):
    A, C, rho, th = _material(case, seed)
    s = {"case": case, "grid": Grid(case, A, C, rho, th)}
    g, kind = s["grid"].h, case["kind"]
    kappas = _kappas(seed, case.get("nk", 1))
    if kind == "bands":
        s["kappas"] = kappas
        s["opt"] = pc.pc_options_default(precision=pc.PC_PREC_MIXED if case["precision"] == "mixed" else pc.PC_PREC_FP64)
        return s
    pc.pc_set_k(g, kappas[0])
    blocks = _blocks(case)
    per = case.get("count", 1) // len(blocks)
    s["x"] = _vectors(case, seed, kappas[0], blocks, per)
    s["sigma"] = _shift(C, rho)
    if kind == "grad":
        s["lam"], s["w"] = _grad_scalars(case, seed)
        n = case["N"] ** 3
        s["dC"] = torch.zeros(21 * n, dtype=torch.float64, device="cuda")
        s["drho"] = torch.zeros(n, dtype=torch.float64, device="cuda")
    else:
        s["y"] = [torch.zeros_like(x) for x in s["x"]]
    return s


def _grad_scalars(case, seed):
    rng = np.random.default_rng(seed + 5)
    return rng.uniform(0.1, 4.0, case["count"]) * 1e7, rng.uniform(-1.0, 1.0, case["count"])


def run(s):
    case, g = s["case"], s["grid"].h
    kind = case["kind"]
    if kind == "apply":
        b = case["block"]
        if b == 4:  # one launch over the four parity blocks
            pc.pc_apply_batch(g, [0, 1, 2, 3], s["x"], s["y"], [s["sigma"]] * 4)
        elif case["count"] == 1:
            pc.pc_block_apply(g, b, s["x"][0], s["y"][0], shift=s["sigma"])
        else:
            pc.pc_block_apply_many(g, b, case["count"], s["x"][0], s["y"][0], shift=s["sigma"])
        return s["y"]
    if kind == "precond":
        pc.pc_block_precond(g, case["block"], s["sigma"], s["x"][0], s["y"][0], fp32_transforms=case["fp32"])
        return s["y"]
    if kind == "pcg":
        pc.pc_shift_invert_pcg(g, case["block"], s["sigma"], s["x"][0], s["y"][0], tol=1e-10)
        return s["y"]
    if kind == "grad":
        s["dC"].zero_()
        s["drho"].zero_()
        pc.pc_eig_grad(g, case["block"], s["x"][0], s["lam"], s["w"], s["dC"], s["drho"])
        return [s["dC"], s["drho"]]
    # the eigenvalues: which of two blocks a value that both hold is credited to is arbitrary
    if case["nk"] == 1:
        return pc.pc_eigs(g, s["kappas"][0], case["nev"], opt=s["opt"])[0]
    return pc.pc_eigs_multi(g, s["kappas"], case["nev"], opt=s["opt"])[0]


def work(case):
    N, kind = case["N"], case["kind"]
    nb = N ** 3 // 4
    m = N ** 3 if case.get("block", 0) < 0 else nb
    elem = 8 if case.get("dtype") == "c64" else 16
    mat = {"phase": 1, "fcc": 4, "nodewise": 176}[case.get("material", "phase")]
    nodes = m * case.get("count", 1)
    if kind == "apply":  # read x and the material, write y; 294 flops of the stencil per node
        return {"bytes": nodes * 6 * elem + (nodes if case["block"] == 4 else m) * mat, "flops": 294 * nodes}
    fft = 2 * 3 * 5 * m * math.log2(max(2, N ** 3 // 4))  # three components, there and back
    if kind == "precond":
        return {"bytes": m * 6 * elem, "flops": fft + 72 * m}
    if kind == "grad":  # strain (about 130 flops) and 21 products per vector and node
        return {"bytes": nodes * 48 + m * 22 * 8, "flops": nodes * (130 + 21 * 6)}
    if kind == "pcg":  # 25 iterations: operator, preconditioner, vector updates
        return {"bytes": 25 * m * 16 * 3 * 12, "flops": 25 * (m * (294 + 72 + 48) + fft)}
    # one shift-invert solve of 25 iterations for every returned pair
    solves = case["nk"] * case["nev"]
    return {"bytes": solves * 25 * nb * 16 * 3 * 12, "flops": solves * 25 * (nb * (294 + 72 + 48) + 2 * 3 * 5 * nb * math.log2(N ** 3 // 4))}


# ---------------------------------------------------------------------------------- 64-bit values
SIGNS = [(1, 1), (1, -1), (-1, 1), (-1, -1)]                # (s2, s3) of the diagonals d_l = (1, s2, s3)
CSL = [(1, 1, 1, 1), (1, 1, -1, -1), (1, -1, 1, -1)]        # reconstruction signs


def _moved(x, d, phi):
    """x(r + d) for d in {-1, 1}^3, Bloch-periodic; x [..., k, j, i]."""
    for axis, step, ph in ((-1, d[0], phi[0]), (-2, d[1], phi[1]), (-3, d[2], phi[2])):
        x = torch.roll(x, -step, dims=axis)
        at = x.shape[axis] - 1 if step > 0 else 0
        x.select(axis, at).mul_(complex(math.cos(ph), step * math.sin(ph)))
    return x


def _strain(x, phi, mix):
    """Six strain components (engineering shear) of x [..., 3, N, N, N]; the factor i is left out."""
    H = [0, 0, 0]
    for l, (s2, s3) in enumerate(SIGNS):
        g = _moved(x, (-1, -s2, -s3), phi) - x
        for s in range(3):
            H[s] = H[s] + CSL[s][l] * g
    G = [sum(mix[s][m] * H[s] for s in range(3)) for m in range(3)]
    G = [[G[m].select(-4, a) for a in range(3)] for m in range(3)]
    return [G[0][0], G[1][1], G[2][2], G[2][1] + G[1][2], G[2][0] + G[0][2], G[1][0] + G[0][1]]


VOIGT = [[0, 5, 4], [5, 1, 3], [4, 3, 2]]


def _operator(x, phi, mix, Cn, rn, shift):
    """(A - shift M) x on the full grid; Cn [6][6] and rn numbers or fields [N, N, N]."""
    e = _strain(x, phi, mix)
    t = [sum(Cn[p][r] * e[r] for r in range(6)) for p in range(6)]
    y = -shift * (rn * x)
    for l, (s2, s3) in enumerate(SIGNS):
        F = 0
        for s in range(3):
            P = torch.stack([sum(mix[s][m] * t[VOIGT[a][m]] for m in range(3)) for a in range(3)], dim=-4)
            F = F + CSL[s][l] * P
        y = y + _moved(F, (1, s2, s3), phi) - F
    return y


def _exact_material(case, seed):
    A, C, rho, th = _material(case, seed)
    N = case["N"]
    L, ainv = _hat(A)
    t = torch.from_numpy(th.astype(np.float64)).cuda().reshape(N, N, N)
    Cn = [[(1 - t) * (C[0][p][r] / C0) + t * (C[1][p][r] / C0) for r in range(6)] for p in range(6)]
    rn = (1 - t) * (rho[0] / RHO0) + t * (rho[1] / RHO0)
    mix = [[float(ainv[s, m]) * N / 4 for m in range(3)] for s in range(3)]
    return A, C, rho, Cn, rn, mix, L


def _embed(x, N, b):
    if b < 0:
        return x.reshape(*x.shape[:-1], N, N, N).to(torch.complex128)
    out = torch.zeros(*x.shape[:-1], N ** 3, dtype=torch.complex128, device="cuda")
    out[..., _block_nodes(N, b)] = x.to(torch.complex128)
    return out.reshape(*x.shape[:-1], N, N, N)


def _extract(x, N, b):
    x = x.reshape(*x.shape[:-3], N ** 3)
    return x if b < 0 else x[..., _block_nodes(N, b)]


def _precond_maker(N, phi, mix, Cref, rref, sigma):
    """r -> (A_ref - sigma rho_ref)^-1 r on the full grid, through the Bloch Fourier symbol."""
    a = [((phi[l] % (2 * math.pi)) + 2 * math.pi * torch.arange(N, device="cuda", dtype=torch.float64)) / N for l in range(3)]
    al = (a[0][None, None, :], a[1][None, :, None], a[2][:, None, None])
    H = [0, 0, 0]
    for l, (s2, s3) in enumerate(SIGNS):
        g = torch.exp(-1j * (al[0] + s2 * al[1] + s3 * al[2])) - 1
        for s in range(3):
            H[s] = H[s] + CSL[s][l] * g
    G = [sum(mix[s][m] * H[s] for s in range(3)) for m in range(3)]
    z = torch.zeros_like(G[0])
    E = [[G[0], z, z], [z, G[1], z], [z, z, G[2]], [z, G[2], G[1]], [G[2], z, G[0]], [G[1], G[0], z]]
    S = [[sum(E[p][u].conj() * (Cref[p][r] * E[r][v]) for p in range(6) for r in range(6)) for v in range(3)] for u in range(3)]
    for u in range(3):
        S[u][u] = S[u][u] - sigma * rref
    cof = [[S[(u + 1) % 3][(v + 1) % 3] * S[(u + 2) % 3][(v + 2) % 3] - S[(u + 1) % 3][(v + 2) % 3] * S[(u + 2) % 3][(v + 1) % 3]
            for v in range(3)] for u in range(3)]
    det = sum(S[0][v] * cof[0][v] for v in range(3))
    F = [[cof[v][u] / det for v in range(3)] for u in range(3)]
    pos = torch.arange(N, device="cuda", dtype=torch.float64) / N
    tw = [torch.exp(1j * (phi[l] % (2 * math.pi)) * pos) for l in range(3)]
    wave = tw[2][:, None, None] * tw[1][None, :, None] * tw[0][None, None, :]

    def solve(r):
        h = torch.fft.fftn(r * wave.conj(), dim=(-3, -2, -1))
        h = torch.stack([sum(F[u][v] * h.select(-4, v) for v in range(3)) for u in range(3)], dim=-4)
        return torch.fft.ifftn(h, dim=(-3, -2, -1)) * wave
    return solve


def exact(case, seed):
    kind, N = case["kind"], case["N"]
    if kind == "bands" and N > NEV_DENSE_N:
        return None  # a dense spectrum of this size takes minutes
    A, C, rho, Cn, rn, mix, L = _exact_material(case, seed)
    kappas = _kappas(seed, case.get("nk", 1))
    phi = [2 * math.pi * float(v) for v in kappas[0]]
    if kind == "bands":
        out = np.stack([_dense(N, [2 * math.pi * float(v) for v in k], mix, Cn, rn, case["nev"]) for k in kappas])
        out = out * C0 / (RHO0 * L * L)
        return out[0] if case["nk"] == 1 else out
    blocks = _blocks(case)
    xs = _vectors(case, seed, kappas[0], blocks, case.get("count", 1) // len(blocks))
    sigma = _shift(C, rho)
    if kind == "apply":
        out = []
        for b, x in zip(blocks, xs):
            out.append(torch.stack([_extract(_operator(_embed(v, N, b), phi, mix, Cn, rn, sigma), N, b) for v in x]))
        return out
    b, x = blocks[0], xs[0]
    if kind == "grad":
        lam, w = _grad_scalars(case, seed)
        dC = torch.zeros(21, N ** 3, dtype=torch.float64, device="cuda")
        dr = torch.zeros(N ** 3, dtype=torch.float64, device="cuda")
        for v in range(case["count"]):
            e = _strain(_embed(x[v], N, b), phi, mix)
            if b >= 0:  # the other blocks' nodes belong to other vectors
                keep = torch.zeros(N ** 3, dtype=torch.float64, device="cuda")
                keep[_block_nodes(N, b)] = 1.0
                e = [f * keep.reshape(N, N, N) for f in e]
            for q, (p, r) in enumerate(zip(*IU)):
                dC[q] += (w[v] / (RHO0 * L * L) * (1 if p == r else 2)) * (e[p].conj() * e[r]).real.reshape(-1)
            dr -= w[v] * lam[v] / RHO0 * _embed(x[v], N, b).abs().square().sum(0).reshape(-1)
        return [dC.reshape(-1), dr]
    Cref = [[float(Cn[p][r].mean()) for r in range(6)] for p in range(6)]
    P = _precond_maker(N, phi, mix, Cref, float(rn.mean()), sigma)
    if kind == "precond":
        return [torch.stack([_extract(P(_embed(v, N, b)), N, b) for v in x])]
    # conjugate gradients to working precision
    r = _embed(x[0], N, b)
    sol, rr0, p, rz = torch.zeros_like(r), r.norm(), None, None
    for _ in range(200):
        z = P(r)
        rz_new = torch.vdot(r.reshape(-1), z.reshape(-1)).real
        p = z if p is None else z + (rz_new / rz) * p
        rz = rz_new
        Ap = _operator(p, phi, mix, Cn, rn, sigma)
        al = rz / torch.vdot(p.reshape(-1), Ap.reshape(-1)).real
        sol = sol + al * p
        r = r - al * Ap
        if float(r.norm()) <= 1e-14 * float(rr0):
            break
    return [torch.stack([_extract(sol, N, b)])]


def _dense(N, phi, mix, Cn, rn, nev):
    """Lowest eigenvalues (hat units) from the dense pencils of the four parity blocks."""
    vals = []
    for b in range(4):
        idx = _block_nodes(N, b)
        m = idx.numel()
        root = rn.reshape(-1)[idx].rsqrt().repeat(3)
        M = torch.empty(3 * m, 3 * m, dtype=torch.complex128, device="cuda")
        step = max(1, 2 ** 21 // N ** 3)
        for c in range(0, 3 * m, step):
            cols = torch.arange(c, min(3 * m, c + step), device="cuda")
            x = torch.zeros(cols.numel(), 3 * m, dtype=torch.complex128, device="cuda")
            x[torch.arange(cols.numel(), device="cuda"), cols] = 1.0
            y = _operator(_embed(x.reshape(-1, 3, m), N, b), phi, mix, Cn, rn, 0.0)
            M[:, cols] = _extract(y, N, b).reshape(cols.numel(), 3 * m).T
        M = root[:, None] * M * root[None, :]
        vals.append(torch.linalg.eigvalsh(0.5 * (M + M.mH)).cpu().numpy())
    return np.sort(np.concatenate(vals))[:nev]
