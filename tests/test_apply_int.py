"""The integer-pipe complex128 apply and the complex64 cell apply (host emulation of their per-thread
functions) against the two-pass apply, over the forms both accept (CPU only).

Tolerance: both sides round at most about 60 times in a chain, and a unit roundoff is 2^-53, so
two correct results differ by at most 2 * 60 * 2^-53 = 1.4e-14 of the output's norm on broad-band
vectors.
"""

import ctypes
import importlib.util
import os

import numpy as np
import pytest

from oracle import oracle as O
from workloads import complex_gaussian, two_phase_sphere

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOL = 1.4e-14
TWO_PASS, INT = 30, 60
LATTICES = {"cubic": np.eye(3), "fcc": 0.5 * (np.ones((3, 3)) - np.eye(3)),
            "skew": np.array([[1.0, 0.2, -0.1], [0.0, 0.9, 0.3], [0.1, 0.0, 1.2]])}


@pytest.fixture(scope="module")
def emu():
    spec = importlib.util.spec_from_file_location(
        "pcband_build", os.path.join(ROOT, "paper_2606_03599_gb300", "build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    lib = ctypes.CDLL(mod.build_emulator())
    dp = ctypes.POINTER(ctypes.c_double)
    lib.pc_emu_apply.argtypes = [ctypes.c_int] * 5 + [dp, dp, dp, ctypes.c_int, dp, ctypes.c_void_p,
                                                      ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p,
                                                      ctypes.c_double]
    lib.pc_emu_apply.restype = ctypes.c_int
    return lib


def both(lib, N, block, lattice, matkind, x, tilings, kappa=(0.21, -0.33, 0.4), shift=0.7):
    """The two-pass result and the integer kernel's for each (shape, tz) of `tilings`."""
    rng = np.random.default_rng(N + matkind)
    n = N ** 3
    cell = two_phase_sphere(N, 0.35, 3)
    A = LATTICES[lattice]
    ainv = np.ascontiguousarray(np.linalg.inv(A / abs(np.linalg.det(A)) ** (1 / 3)))
    idx = np.arange(n) if block < 0 else O.block_index((N,) * 3, block)
    C, rho = cell.C / 1e9, cell.rho / 1e3
    if matkind == 2:
        iu = np.triu_indices(6)
        G = rng.standard_normal((n, 6, 6))
        Cn = C[cell.phase.astype(int)] + 0.1 * (G + np.transpose(G, (0, 2, 1)))
        q2 = (N / 4.0) ** 2 if lattice == "cubic" else 1.0
        lay = np.concatenate([Cn[:, iu[0], iu[1]].T * q2, rng.uniform(1, 8, (1, n))], axis=0)
        mat = np.ascontiguousarray(lay[:, idx])
    elif matkind == 1:
        mat = rng.uniform(0, 1, n).astype(np.float32)
        mat[:2] = [0.0, 1.0]
        mat = np.ascontiguousarray(mat[idx])
    else:
        mat = np.ascontiguousarray(cell.phase[idx])
    dp = ctypes.POINTER(ctypes.c_double)
    C72 = np.ascontiguousarray(C.reshape(72))
    phi = np.ascontiguousarray(2 * np.pi * (np.asarray(kappa) - np.floor(kappa)))
    x = np.ascontiguousarray(x[:, idx])
    out = []
    for shape, tz in [(TWO_PASS, 0)] + list(tilings):
        y = np.full_like(x, np.nan)
        assert lib.pc_emu_apply(N, block, 1 if x.dtype == np.complex64 else 2, shape, tz, C72.ctypes.data_as(dp), rho.ctypes.data_as(dp),
                                ainv.ctypes.data_as(dp), int(lattice == "cubic"), phi.ctypes.data_as(dp),
                                mat.ctypes.data, matkind, x.ctypes.data, y.ctypes.data, shift) == 0
        out.append(y)
    return out


# (shape, planes per CTA): the default tile whole and cut, and tiles that leave ragged edges
TILINGS = [(INT, 0), (INT, 3), (6033, 2), (6052, 5), (6119, 4), (6219, 1)]


@pytest.mark.parametrize("N", [4, 6, 8, 14, 34])
@pytest.mark.parametrize("lattice", list(LATTICES))
@pytest.mark.parametrize("matkind", [0, 1, 2])
@pytest.mark.parametrize("block", [-1, 1, 2])
def test_integer_apply_equals_two_pass(emu, N, lattice, matkind, block):
    if N == 34 and (block != 2 or lattice == "skew"):
        pytest.skip("one block and two lattices at the largest size")
    ref, *got = both(emu, N, block, lattice, matkind, complex_gaussian((3, N ** 3), 7), TILINGS)
    for y in got:
        assert np.linalg.norm(y - ref) <= TOL * np.linalg.norm(ref)
        assert np.array_equal(y, got[0])  # a node's arithmetic does not depend on the tile


@pytest.mark.parametrize("N", [4, 6, 8, 14, 34])
@pytest.mark.parametrize("lattice", ["cubic", "skew"])
@pytest.mark.parametrize("matkind", [0, 1])
@pytest.mark.parametrize("block", [-1, 1, 2])
def test_cell_apply_equals_two_pass_in_complex64(emu, N, lattice, matkind, block):
    """The complex64 cell kernel against the two-pass kernels in complex64: the same operations in
    nearly the same order, so at most 2 * 60 roundings of 2^-24 apart."""
    if N == 34 and (block != 2 or lattice == "skew"):
        pytest.skip("one block and one lattice at the largest size")
    x = complex_gaussian((3, N ** 3), 7).astype(np.complex64)
    ref, *got = both(emu, N, block, lattice, matkind, x, TILINGS)
    for y in got:
        assert np.linalg.norm(y - ref) <= 120 * 2.0 ** -24 * np.linalg.norm(ref)
        assert np.array_equal(y, got[0])


@pytest.mark.parametrize("lattice,matkind", [("cubic", 0), ("fcc", 1), ("cubic", 2)])
@pytest.mark.parametrize("value", [0.0, 5e-324, 1e-300, 1e-200, 1e250, 1e300, np.inf, np.nan])
def test_integer_apply_takes_every_double(emu, lattice, matkind, value):
    """Nodes outside the exponent range go through FP64: infinities and NaN spread as they do there,
    and huge or tiny values keep their relative accuracy."""
    N, block = 8, 3
    x = complex_gaussian((3, N ** 3), 9)
    if value == 0.0:
        x[:] = 0.0
    elif np.isfinite(value):
        x *= value
    else:
        x[1, O.block_index((N,) * 3, block)[37]] = value
    ref, y, cut = both(emu, N, block, lattice, matkind, x, [(INT, 0), (6023, 3)])
    fine = np.isfinite(ref)
    for v in (y, cut):
        assert np.array_equal(fine, np.isfinite(v))
        scale = np.abs(ref[fine]).max(initial=0.0)
        assert np.abs(v[fine] - ref[fine]).max(initial=0.0) <= max(TOL * 4 * scale, 1e-320)


def test_integer_apply_keeps_each_nodes_own_scale(emu):
    """A vector whose size falls by 1e-60 across the cell: every node's output is accurate relative
    to the values around it, not to the vector's largest."""
    N, block = 16, 0
    l = np.arange(N ** 3)
    x = complex_gaussian((3, N ** 3), 4) * 10.0 ** (-4.0 * (l // (N * N)))
    ref, y = both(emu, N, block, "cubic", 0, x, [(INT, 5)], kappa=(0.2, 0.1, 0.3))
    scale = np.abs(ref).reshape(3, N, -1).max(axis=(0, 2))[None, :, None]
    assert (np.abs(y - ref).reshape(3, N, -1) <= 4 * TOL * scale).all()


@pytest.mark.parametrize("n", [1, 4, 8])
@pytest.mark.parametrize("spread", [0, 12, 60])
@pytest.mark.parametrize("scale", [1e-100, 1.0, 1e100])
def test_limb_group_sum(emu, n, spread, scale):
    """The group products of the outer loop against extended precision.  A value is cut at 2^-57 of
    its group's largest and a product drops its low x low part, at most 2^-56 of the largest
    product, so each of the 2 n real products is off by at most 3 * 2^-56 of it; the conversion to a
    double adds half a unit of the result and of the group's unit."""
    dp = ctypes.POINTER(ctypes.c_double)
    emu.pc_emu_limb_dot.argtypes = [ctypes.c_int, dp, dp, dp]
    rng = np.random.default_rng(n + spread)
    for _ in range(50):
        a, b = (rng.standard_normal((n, 2)) * 2.0 ** -rng.integers(0, spread + 1, (n, 2)) for _ in range(2))
        a *= scale
        a[rng.random((n, 2)) < 0.1] = 0.0
        a[0, 0] = scale
        out = np.zeros(2)
        assert emu.pc_emu_limb_dot(n, a.ctypes.data_as(dp), b.ctypes.data_as(dp), out.ctypes.data_as(dp)) == 0
        x, y = a.astype(np.longdouble), b.astype(np.longdouble)
        ref = np.array([(x[:, 0] * y[:, 0] - x[:, 1] * y[:, 1]).sum(), (x[:, 0] * y[:, 1] + x[:, 1] * y[:, 0]).sum()])
        top = np.abs(a).max() * np.abs(b).max()
        assert (np.abs(out - ref) <= (2 * n * 3 + 2) * 2.0 ** -56 * top * 4 + 2.0 ** -53 * np.abs(ref)).all()


@pytest.mark.parametrize("value", [np.inf, np.nan, 1e-250, 1e250])
def test_limb_group_leaves_extreme_values_to_fp64(emu, value):
    dp = ctypes.POINTER(ctypes.c_double)
    a = np.full((2, 2), value)
    b = np.ones((2, 2))
    out = np.zeros(2)
    for u, v in ((a, b), (b, a)):
        assert emu.pc_emu_limb_dot(2, u.ctypes.data_as(dp), v.ctypes.data_as(dp), out.ctypes.data_as(dp)) == 1
