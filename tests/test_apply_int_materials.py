"""The integer-pipe complex128 apply on nodewise materials that a design field holds: voids and tables far
from the usual moduli (host emulation, CPU only).

Tolerance: as tests/test_apply_int.py, two results of at most 60 roundings of 2^-53 each, 1.4e-14 of the
output's norm.
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


@pytest.fixture(scope="module")
def emu():
    spec = importlib.util.spec_from_file_location(
        "pcband_build", os.path.join(ROOT, "paper_2606_03599_gb300", "build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return ctypes.CDLL(mod.build_emulator())


def nodewise_apply(lib, N, block, scale, shift=0.7):
    """Two-pass result, integer result and columns handed to FP64, for the sphere cell's nodewise table with
    every node's stiffness times scale[node]."""
    cell = two_phase_sphere(N, 0.35, 3)
    idx = np.arange(N ** 3) if block < 0 else O.block_index((N,) * 3, block)
    iu = np.triu_indices(6)
    C = (cell.C / 1e9)[cell.phase.astype(int)][:, iu[0], iu[1]] * scale[:, None]
    rho = np.where(cell.phase != 0, cell.rho[1], cell.rho[0]) / 1e3
    mat = np.ascontiguousarray(np.concatenate([C.T * (N / 4.0) ** 2, rho[None]], axis=0)[:, idx])
    x = np.ascontiguousarray(complex_gaussian((3, N ** 3), 11)[:, idx])
    C72, two, ainv = np.zeros(72), np.ones(2), np.eye(3).reshape(9).copy()
    phi = 2 * np.pi * np.array([0.21, 0.67, 0.4])
    vp = ctypes.c_void_p
    out = []
    for shape in (TWO_PASS, INT):
        y = np.full_like(x, np.nan)
        assert lib.pc_emu_apply(N, block, 2, shape, 0, vp(C72.ctypes.data), vp(two.ctypes.data), vp(ainv.ctypes.data), 1,
                                vp(phi.ctypes.data), vp(mat.ctypes.data), 2, vp(x.ctypes.data), vp(y.ctypes.data),
                                ctypes.c_double(shift)) == 0
        out.append(y)
    return out[0], out[1], lib.pc_emu_slow_columns()


@pytest.mark.parametrize("block", [-1, 2])
@pytest.mark.parametrize("void", ["half", "all", "scattered"])
def test_void_nodes_have_no_flux_and_stay_on_the_fast_path(emu, block, void):
    """A node of zero stiffness (pc_grid_create_nodewise takes it) has zero fluxes; no column is handed to
    the per-thread FP64 path for it."""
    N = 12
    k = np.arange(N ** 3) // (N * N)
    scale = {"half": (k < N // 2) * 1.0, "all": np.zeros(N ** 3),
             "scattered": (np.random.default_rng(1).random(N ** 3) < 0.8) * 1.0}[void]
    ref, y, slow = nodewise_apply(emu, N, block, scale)
    assert slow == 0
    assert np.linalg.norm(y - ref) <= TOL * np.linalg.norm(ref)
