"""The fixed-point interface offsets of PPM and PPM-EP (csrc/mhd_fixed.cuh), compiled for the host, against
exact rational arithmetic: random windows, exponent gaps around the clamps, ties, zeros, deep
cancellation, and the ends of the exponent range."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "mhd_fixed.cuh"
extern "C" void ppm(const unsigned long long* w, unsigned long long* o, long n) {
  for (long i = 0; i < n; ++i) mhd::ppm_split_bits(w[3 * i], w[3 * i + 1], w[3 * i + 2], o[2 * i], o[2 * i + 1]);
}
extern "C" void ppm_ep(const unsigned long long* w, unsigned long long* o, long n) {
  for (long i = 0; i < n; ++i) {
    const unsigned long long* b = w + 3 * i;
    int e[3], m = 0;
    for (int k = 0; k < 3; ++k) { e[k] = (int)(b[k] >> 52) & 0x7ff; m = e[k] > m ? e[k] : m; }
    mhd::ppm_ep_split_bits(b[0], b[1], b[2], m, e[0], e[1], e[2], o[2 * i], o[2 * i + 1]);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    (d / "f.cpp").write_text(SRC)
    so = str(d / "f.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                           os.path.join(ROOT, "paper_2609_10816_gb300", "csrc"), "-o", so, str(d / "f.cpp")])
    return ctypes.CDLL(so)


def _offsets(f, w):
    w = np.ascontiguousarray(w, dtype=np.float64)
    o = np.zeros((len(w), 2))
    p = ctypes.POINTER(ctypes.c_ulonglong)
    f(w.view(np.uint64).ctypes.data_as(p), o.view(np.uint64).ctypes.data_as(p), ctypes.c_long(len(w)))
    return o


def _field(lo, hi, rng, n):
    """doubles of either sign with exponent fields in [lo, hi], some of few significant bits"""
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    few = rng.random(n) < 0.3
    m = np.where(few, m & np.uint64(0xF << 48), m)
    e = rng.integers(lo, hi + 1, n).astype(np.uint64)
    return (m | (e << np.uint64(52)) | (rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63))).view(np.float64)


def _windows(kind, rng, n):
    """(dl, d, dn)"""
    if kind == "random":
        return rng.normal(size=(n, 3))
    if kind == "smooth":  # nearly equal differences: dl - dn cancels
        d = rng.normal(size=n)
        return d[:, None] * (1.0 + 10.0 ** rng.uniform(-16, -1, (n, 1)) * rng.normal(size=(n, 3)))
    if kind == "gaps":  # binades apart around the clamps (2^3 above, 2^-63 below) and beyond
        d = _field(600, 1400, rng, n)
        g = rng.choice([-4, -3, -2, -1, 0, 1, 2, 3, 4, 5, 53, 59, 60, 61, 62, 63, 64, 65, 200], (n, 2))
        side = _field(1023, 1023, rng, 2 * n).reshape(n, 2) * 2.0 ** g * np.abs(d)[:, None]
        return np.stack([side[:, 0], d, side[:, 1]], axis=1)
    if kind == "ends":  # the ends of the range of exponent fields, with neighbours outside it
        e = rng.choice([128, 129, 130, 2037, 2038, 2039], n)
        d = np.array([_field(x, x, rng, 1)[0] for x in e])
        lo = np.array([_field(max(1, x - 127), x, rng, 1)[0] for x in e])
        hi = np.array([_field(max(1, x - 3), x, rng, 1)[0] for x in e])
        return np.stack([lo, d, hi], axis=1)
    if kind == "few bits":
        w = rng.integers(-6, 7, (n, 3)).astype(float)
        w[:, 1] = np.where(w[:, 1] == 0, 1.0, w[:, 1])
        return w
    # the fourth-order value on or next to a cell's value: d/2 + (dl - dn)/12 is zero or one bit of d
    d = rng.integers(1, 1 << 20, n).astype(float)
    dl = rng.integers(1, 1 << 20, n).astype(float)
    return np.stack([dl, d, dl + 6.0 * d + rng.integers(-1, 2, n) * 2.0**-20], axis=1)


KINDS = ("random", "smooth", "gaps", "ends", "few bits", "ties")


def _slope2(a, d):
    """the doubled limited slope of differences a, d"""
    if a == 0 or d == 0 or (a > 0) != (d > 0):
        return Fraction(0)
    m = min(abs(a + d), 4 * abs(a), 4 * abs(d))
    return m if d > 0 else -m


@pytest.mark.parametrize("kind", KINDS)
def test_ppm(lib, kind):
    w = _windows(kind, np.random.default_rng(3), 4000)
    o = _offsets(lib.ppm, w)
    for (dl, d, dn), (r, s) in zip(w.tolist(), o.tolist()):
        dl, d, dn = Fraction(dl), Fraction(d), Fraction(dn)
        x = d / 2 + (_slope2(dl, d) - _slope2(d, dn)) / 12
        # one rounding to nearest, and a sixteenth of its unit for the bits cut off
        assert abs(Fraction(r) - x) <= Fraction(9, 8) * Fraction(1, 1 << 53) * abs(x)
        assert abs(Fraction(s) - (d - x)) <= Fraction(9, 8) * Fraction(1, 1 << 53) * abs(d - x)


def test_ppm_of_a_zero_difference(lib):
    for z in (0.0, -0.0):
        o = _offsets(lib.ppm, [[1.0, z, 2.0], [0.0, z, -0.0], [-1e300, z, 5e-324]])
        assert (o == 0.0).all()


@pytest.mark.parametrize("kind", KINDS)
def test_ppm_ep(lib, kind):
    w = _windows(kind, np.random.default_rng(4), 4000)
    if kind == "gaps":  # (the largest of the three differences sets the scale)
        w = w[np.abs(w).max(axis=1) < 2.0**1016]
    o = _offsets(lib.ppm_ep, w)
    for (dl, d, dn), (r, s) in zip(w.tolist(), o.tolist()):
        big = max(abs(dl), abs(d), abs(dn))
        dl, d, dn = Fraction(dl), Fraction(d), Fraction(dn)
        x = d / 2 + (dl - dn) / 12
        # half a unit of the last place of the result, and 5 units of the common scale (three differences cut
        # off, the division's 3), of which the largest difference has at least 2^59
        cut = Fraction(5, 1 << 59) * Fraction(big)
        assert abs(Fraction(r) - x) <= Fraction(1, 1 << 53) * (abs(x) + cut) + cut
        assert abs(Fraction(s) - (d - x)) <= Fraction(1, 1 << 53) * (abs(d - x) + cut) + cut
