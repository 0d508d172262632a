"""The integer-pipe complex128 apply keeps FP64's accuracy on every kind of vector and material, not only on
broad-band ones (host emulation of its per-thread functions, CPU only).

Both it and the two-pass FP64 apply are compared with the operator in extended precision, for each
component and each of the real and imaginary parts by itself.

Tolerance: the integer result may be as far off as the FP64 one, plus one rounding of the result (2^-53, as
FP64's own error vanishes on some inputs), plus what the reference itself can tell: its 64-bit significands
carry 60 roundings of 2^-64 of the fluxes, and a long wave's output is (2 pi / N)^2 / 8 of those.
"""

import ctypes
import importlib.util
import os

import numpy as np
import pytest

from oracle import oracle as O

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LD, CLD = np.longdouble, np.clongdouble
IU = np.triu_indices(6)
LATTICES = {"cubic": np.eye(3), "fcc": 0.5 * (np.ones((3, 3)) - np.eye(3)),
            "skew": np.array([[1.0, 0.2, -0.1], [0.0, 0.9, 0.3], [0.1, 0.0, 1.2]])}
SIGNS = [(1, 1), (1, -1), (-1, 1), (-1, -1)]
CSL = [(1, 1, 1, 1), (1, 1, -1, -1), (1, -1, 1, -1)]
VOIGT = [[0, 5, 4], [5, 1, 3], [4, 3, 2]]


@pytest.fixture(scope="module")
def emu():
    spec = importlib.util.spec_from_file_location(
        "pcband_build", os.path.join(ROOT, "paper_2606_03599_gb300", "build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return ctypes.CDLL(mod.build_emulator())


def isotropic(K, G):
    C = np.zeros((6, 6))
    C[:3, :3] = K - 2 * G / 3
    C[range(3), range(3)] = K + 4 * G / 3
    C[range(3, 6), range(3, 6)] = G
    return C


def moved(x, d, phi):
    for axis, step, ph in ((-1, d[0], phi[0]), (-2, d[1], phi[1]), (-3, d[2], phi[2])):
        x = np.roll(x, -step, axis=axis)
        at = [slice(None)] * x.ndim
        at[axis] = x.shape[axis] - 1 if step > 0 else 0
        x[tuple(at)] *= CLD(complex(np.cos(ph), step * np.sin(ph)))
    return x


def reference(x, N, phi, mix, C, rho, shift):
    """(A - shift M) x on the full grid in extended precision; C [6][6] and rho numbers or fields."""
    x = x.reshape(3, N, N, N).astype(CLD)
    H = [0, 0, 0]
    for l, (s2, s3) in enumerate(SIGNS):
        g = moved(x, (-1, -s2, -s3), phi) - x
        for s in range(3):
            H[s] = H[s] + CSL[s][l] * g
    G = [sum(LD(mix[s][m]) * H[s] for s in range(3)) for m in range(3)]
    e = [G[0][0], G[1][1], G[2][2], G[2][1] + G[1][2], G[2][0] + G[0][2], G[1][0] + G[0][1]]
    t = [sum(C[p][r] * e[r] for r in range(6)) for p in range(6)]
    y = -LD(shift) * (rho * x)
    for l, (s2, s3) in enumerate(SIGNS):
        F = 0
        for s in range(3):
            F = F + CSL[s][l] * np.stack([sum(LD(mix[s][m]) * t[VOIGT[a][m]] for m in range(3)) for a in range(3)])
        y = y + moved(F, (1, s2, s3), phi) - F
    return y.reshape(3, -1)


def three(lib, N, lattice, kind, C, rho, theta, x, kappa, shift=0.0, block=-1):
    """Extended, two-pass and integer results.  kind: 0 phase ids, 1 fractions, 2 the same mixture node by node."""
    A = LATTICES[lattice]
    cubic = lattice == "cubic"
    ainv = np.ascontiguousarray(np.linalg.inv(A / abs(np.linalg.det(A)) ** (1 / 3)))
    phi = np.ascontiguousarray(2 * np.pi * (np.asarray(kappa, float) - np.floor(kappa)))
    n = N ** 3
    idx = np.arange(n) if block < 0 else O.block_index((N,) * 3, block)
    th = np.asarray(theta, float)
    if kind == 2:
        c21 = (1 - th)[:, None] * C[0][IU] + th[:, None] * C[1][IU]
        rn = (1 - th) * rho[0] + th * rho[1]
        mat = np.ascontiguousarray(np.concatenate([c21.T * ((N / 4.0) ** 2 if cubic else 1.0), rn[None]])[:, idx])
        Cx = [[None] * 6 for _ in range(6)]
        for q, (p, r) in enumerate(zip(*IU)):
            Cx[p][r] = Cx[r][p] = c21[:, q].astype(LD).reshape(N, N, N)
        rx = rn.astype(LD).reshape(N, N, N)
    else:
        mat = np.ascontiguousarray(np.asarray(theta, np.uint8 if kind == 0 else np.float32)[idx])
        t = th.astype(np.float32).astype(LD).reshape(N, N, N)
        Cx = [[(1 - t) * LD(C[0][p][r]) + t * LD(C[1][p][r]) for r in range(6)] for p in range(6)]
        rx = (1 - t) * LD(rho[0]) + t * LD(rho[1])
    mix = [[(N / 4 if s == m else 0) if cubic else ainv[s, m] * N / 4 for m in range(3)] for s in range(3)]
    full = np.zeros((3, n), complex)
    full[:, idx] = x[:, idx]
    out = [reference(full, N, phi, mix, Cx, rx, shift)[:, idx]]
    C72, rh = np.ascontiguousarray(np.reshape(C, 72)), np.ascontiguousarray(rho, float)
    xb = np.ascontiguousarray(x[:, idx])
    vp = ctypes.c_void_p
    # fractions far apart are measured against what the FP64 kernels blend
    for shape in (30, 60):
        y = np.full_like(xb, np.nan)
        assert lib.pc_emu_apply(N, block, 2, shape, 0, vp(C72.ctypes.data), vp(rh.ctypes.data), vp(ainv.ctypes.data),
                                int(cubic), vp(phi.ctypes.data), vp(mat.ctypes.data), kind, vp(xb.ctypes.data),
                                vp(y.ctypes.data), ctypes.c_double(shift)) == 0
        out.append(y)
    return out


def parts(y):
    return np.concatenate([y.real, y.imag])


def check(ref, fp64, got, N, where=slice(None)):
    r, f, g = (parts(v)[:, where] for v in (ref, fp64, got))
    norm = lambda v: np.sqrt((v.astype(LD) ** 2).sum(axis=1))
    told = 60 * 2.0 ** -64 * 8 / (2 * np.pi / N) ** 2 * np.sqrt((r ** 2).sum())
    for err, most in zip(norm(g - r), norm(f - r) + 2.0 ** -53 * norm(r) + told):
        assert err <= most, (err, most)


def wave(N, q, pol):
    p = np.arange(N) / N
    w = np.exp(2j * np.pi * (q[2] * p[:, None, None] + q[1] * p[None, :, None] + q[0] * p[None, None, :]))
    return np.asarray(pol, complex)[:, None] * w.reshape(-1)[None]


RHO = [7.8, 2.7]
SOLIDS = {"steel": (160.0, 80.0), "rubber": (1.0, 5e-4), "gel": (1.0, 1e-5), "fluid": (2.2, 0.0)}


@pytest.mark.parametrize("solid", ["steel", "rubber", "gel"])
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("shift", [0.0, -0.3])
def test_transverse_wave_along_an_axis(emu, solid, kind, shift):
    N = 32
    C = isotropic(*SOLIDS[solid])
    x = wave(N, (0.25, 0, 0), (0, 1, 0))
    check(*three(emu, N, "cubic", kind, [C, C], RHO, np.zeros(N ** 3), x, (0.25, 0, 0), shift), N)


@pytest.mark.parametrize("solid", list(SOLIDS))
@pytest.mark.parametrize("lattice", list(LATTICES))
@pytest.mark.parametrize("kind", [0, 1, 2])
def test_waves_off_the_axes(emu, solid, lattice, kind):
    N = 16
    C = isotropic(*SOLIDS[solid])
    x = wave(N, (0.2, 1.1, 0.3), (0.3, 1.0, -0.2)) + 0.1 * wave(N, (1.2, 0.1, 0.3), (1.0, 0.1, 0.5))
    check(*three(emu, N, lattice, kind, [C, C], RHO, np.zeros(N ** 3), x, (0.2, 0.1, 0.3)), N)


def anisotropic(seed):
    rng = np.random.default_rng(seed)
    Q, _ = np.linalg.qr(rng.standard_normal((6, 6)))
    return (Q * rng.uniform(20, 200, 6)) @ Q.T


@pytest.mark.parametrize("small", [1e-5, 1e-8, 1e-12])
@pytest.mark.parametrize("what", ["imag", "component", "uniform", "plane"])
@pytest.mark.parametrize("lattice,kind", [("cubic", 0), ("cubic", 1), ("cubic", 2), ("fcc", 0), ("skew", 1)])
def test_small_next_to_large(emu, small, what, lattice, kind):
    """A small imaginary part, a small component, a small wave on a uniform displacement of another
    component, and a vector that falls from plane to plane."""
    N = 12
    rng = np.random.default_rng(5)
    real = lambda: rng.standard_normal((3, N ** 3))
    kappa = (0.2, 0.1, 0.3)
    C = [isotropic(160, 80), anisotropic(1)]
    C = [0.5 * (c + c.T) for c in C]
    theta = (rng.random(N ** 3) < 0.4) * 1.0
    if what == "imag":
        x, kappa = real() + 1j * small * real(), (0, 0, 0)
    elif what == "component":
        x = real() + 1j * real()
        x[2] *= small
    elif what == "uniform":
        x, kappa = np.ones((3, N ** 3), complex), (0, 0, 0)
        x[1] = small * wave(N, (1, 0, 0), (0, 1, 0))[1]
        theta[:] = 0
    else:
        x = (real() + 1j * real()) * small ** (np.arange(N ** 3) // (N * N) / N)
    check(*three(emu, N, lattice, kind, C, RHO, theta, x, kappa), N)


@pytest.mark.parametrize("contrast", [1e-2, 1e-4, 1e-6, 1e-9])
@pytest.mark.parametrize("lattice", ["cubic", "fcc"])
@pytest.mark.parametrize("kind", [0, 1, 2])
@pytest.mark.parametrize("soft", [0, 1])
def test_soft_phase_on_its_own_scale(emu, contrast, lattice, kind, soft):
    """Nodes deep in the soft one of two phases, held to their own outputs' norm."""
    N, block = 12, 1
    k = np.arange(N ** 3) // (N * N)
    theta = ((k >= 1) & (k < 7)) * 1.0
    hard = 0.5 * (anisotropic(2) + anisotropic(2).T)
    C = [hard * (contrast if soft == p else 1.0) for p in (0, 1)]
    rng = np.random.default_rng(6)
    x = rng.standard_normal((3, N ** 3)) + 1j * rng.standard_normal((3, N ** 3))
    ref, fp64, got = three(emu, N, lattice, kind, C, RHO, theta, x, (0.2, 0.1, 0.3), block=block)
    kb = k[O.block_index((N,) * 3, block)]
    check(ref, fp64, got, N, where=(kb >= 3) & (kb < 5) if soft else (kb >= 9) & (kb < 11))


@pytest.mark.parametrize("entry", [(3, 3), (0, 1), (2, 4)])
@pytest.mark.parametrize("size", [0.0, 1e-7])
@pytest.mark.parametrize("kind", [0, 1, 2])
def test_small_and_zero_stiffness_entries(emu, entry, size, kind):
    """One entry (a shear modulus, a Poisson coupling, a normal-shear coupling) far below the others, on a vector
    whose strain it alone turns into stress."""
    N = 12
    C = isotropic(100, 40)
    C[entry] = C[entry[::-1]] = size
    x = wave(N, (0, 0.25, 0.25), (0, 1, 1)) + 1e-6 * wave(N, (1, 0.25, 0.25), (1, 0, 0))
    check(*three(emu, N, "cubic", kind, [C, C], RHO, np.zeros(N ** 3), x, (0, 0.25, 0.25)), N)


@pytest.mark.parametrize("scale", [1e-280, 1e-150, 1e150, 1e280])
@pytest.mark.parametrize("kind", [0, 2])
def test_extreme_stiffness_and_vector_scales(emu, scale, kind):
    """Stiffness tables and vectors far from hat units, zeros and subnormal values among them: no column leaves
    the fast path."""
    N, block = 8, 2
    rng = np.random.default_rng(8)
    x = (rng.standard_normal((3, N ** 3)) + 1j * rng.standard_normal((3, N ** 3))) * scale
    x[0, ::7] = 5e-324
    x[:, 3::11] = 0.0
    C = [isotropic(160, 80) / scale, isotropic(70, 30) / scale]
    theta = (rng.random(N ** 3) < 0.4) * 1.0
    out = three(emu, N, "cubic", kind, C, RHO, theta, x, (0.2, 0.1, 0.3), block=block)
    assert emu.pc_emu_slow_columns() == 0
    check(*out, N)
