"""The Gram products' sums of complex products on the integer pipe (host emulation of one group of eight, CPU only)
are no further from extended precision than FP64 fused multiply-adds: no bias in squared norms or in sums with real
coefficients, and no loss of small parts or values next to large ones of the same group.

Tolerances.  A product is rounded to three bits below a unit of 2^-58 of the group's largest one, 16 of them, and the sum
is rounded once: 16 * 2^-56 of the largest product + 2^-53 of the result.  In the mean over n groups roundings
cancel: 6 standard deviations of n roundings of rms 2^-54 / sqrt(3) of the result.
"""

import ctypes
import importlib.util
import os

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LD = np.longdouble


@pytest.fixture(scope="module")
def group():
    spec = importlib.util.spec_from_file_location(
        "pcband_build", os.path.join(ROOT, "paper_2606_03599_gb300", "build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    lib = ctypes.CDLL(mod.build_emulator())

    def dot(a, b):
        out = np.zeros(2)
        assert lib.pc_emu_limb_dot(len(a), ctypes.c_void_p(a.ctypes.data), ctypes.c_void_p(b.ctypes.data),
                                   ctypes.c_void_p(out.ctypes.data)) == 0
        return out
    return dot


def exact(a, b):
    ar, ai, br, bi = (v.astype(LD) for v in (a.real, a.imag, b.real, b.imag))
    return np.array([(ar * br - ai * bi).sum(), (ar * bi + ai * br).sum()])


def products(a, b):
    """Largest real product that enters the sum's real and imaginary part."""
    rr = np.maximum(np.abs(a.real * b.real), np.abs(a.imag * b.imag)).max()
    ri = np.maximum(np.abs(a.real * b.imag), np.abs(a.imag * b.real)).max()
    return np.array([rr, ri])


@pytest.mark.parametrize("small", [1.0, 1e-4, 1e-8, 1e-12])
@pytest.mark.parametrize("what", ["imag", "values", "turned", "decay"])
def test_a_group_is_accurate_next_to_its_own_products(group, small, what):
    rng = np.random.default_rng(3)
    for _ in range(100):
        a, b = (rng.standard_normal(8) + 1j * rng.standard_normal(8) for _ in range(2))
        if what == "imag":
            a, b = a.real + 1j * small * a.imag, b.real + 1j * small * b.imag
        elif what == "values":  # large where the other is small
            big = rng.random(8) < 0.5
            a, b = a * np.where(big, 1, small), b * np.where(big, small, 1)
        elif what == "turned":
            a, b = a.real + 1j * small * a.imag, small * b.real + 1j * b.imag
        else:
            a, b = a * small ** (np.arange(8) / 7), b * small ** (np.arange(8)[::-1] / 7)
        err = np.abs(group(a, b) - exact(a, b))
        assert (err <= 16 * 2.0 ** -56 * products(a, b) + 2.0 ** -53 * np.abs(exact(a, b))).all()


def test_squared_norms_have_no_bias(group):
    rng = np.random.default_rng(4)
    n = 4000
    rel = []
    for _ in range(n):
        a = rng.standard_normal(8) + 1j * rng.standard_normal(8)
        ref = exact(a, np.conj(a))[0]
        rel.append(float((group(a, np.conj(a))[0] - ref) / ref))
    assert abs(np.mean(rel)) <= 6 * 2.0 ** -54 / np.sqrt(3 * n)


def test_every_low_half_of_a_factor(group):
    """Values whose significand ends in 2^22: the low half of such a factor is -2^31, in each place of a product."""
    rng = np.random.default_rng(5)
    for k in range(64):
        a, b = (rng.standard_normal(8) + 1j * rng.standard_normal(8) for _ in range(2))
        for v, at in ((a, 1), (b, 2)):
            bits = v.view(np.int64)
            for part in range(16):
                if (k >> (part % 6)) & at or rng.random() < 0.3:
                    bits[part] = (bits[part] & ~0x7fffff) | 0x400000
        err = np.abs(group(a, b) - exact(a, b))
        assert (err <= 16 * 2.0 ** -56 * products(a, b) + 2.0 ** -53 * np.abs(exact(a, b))).all()


@pytest.mark.parametrize("turn", [1, 1j, -1, -1j])
def test_sums_with_real_coefficients_have_no_offset(group, turn):
    """An update with real (or imaginary) coefficients meets one product of each pair only: its roundings have no sign
    in common either."""
    rng = np.random.default_rng(6)
    n, off = 4000, []
    for _ in range(n):
        a = rng.standard_normal(8) + 1j * rng.standard_normal(8)
        b = rng.uniform(0.5, 1.0, 8) * complex(turn)
        off.append(((group(a, b) - exact(a, b)) / np.maximum(products(a, b), 1e-300)).astype(float))
    # rms of a group: 16 roundings of 2^-55 / sqrt(12) and one of the result, below 8 products, of 2^-53 / sqrt(12)
    assert (np.abs(np.mean(off, axis=0)) <= 6 * 8 * 2.0 ** -53 / np.sqrt(12 * n)).all()
