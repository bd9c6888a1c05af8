"""The fixed-point arithmetic of the FP64 stencil on the host (fxmath.h, no GPU) against _Float128.

Bounds (derived in fxmath.h): any element is within 60 units of the integers (2^-57 of the power of
two above the largest neighbour component) of the exact hop sum, plus one FP64 rounding.  An element
that the guard keeps has, in every component it forms, a hop product of 2^53 units or more, so its error
is below 60 of 2^-53 times the sum of the component's terms, plus that rounding: 61.
"""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OUT = os.path.join(ROOT, "tests", "shim", "_build")


@pytest.fixture(scope="module")
def lib():
    os.makedirs(OUT, exist_ok=True)
    so = os.path.join(OUT, "libfxmath_shim.so")
    src = os.path.join(ROOT, "tests", "shim", "fxmath_shim.cpp")
    header = os.path.join(ROOT, "paper_0707_0131_gb300", "csrc", "fxmath.h")
    if not os.path.exists(so) or any(os.path.getmtime(s) > os.path.getmtime(so) for s in (src, header)):
        subprocess.run(["g++", "-O2", "-std=gnu++17", "-fPIC", "-shared", "-o", so, src], check=True)
    L = ctypes.CDLL(so)
    P = ctypes.POINTER(ctypes.c_double)
    for name, args, res in [("fx_to_fixed", [ctypes.c_double, ctypes.c_int], ctypes.c_longlong),
                            ("fx_to_double", [ctypes.c_longlong, ctypes.c_int], ctypes.c_double),
                            ("fx_align", [ctypes.c_longlong, ctypes.c_int], ctypes.c_longlong),
                            ("fx_limbs", [ctypes.c_longlong], ctypes.c_longlong),
                            ("fx_element", [P, P, ctypes.c_int, P, P], ctypes.c_int),
                            ("fx_link_scale", [ctypes.c_double, ctypes.c_double, ctypes.POINTER(ctypes.c_int)], ctypes.c_int)]:
        f = getattr(L, name)
        f.argtypes, f.restype = args, res
    return L


def test_conversions(lib):
    """to_fixed and align within half a unit, limbs exact, to_double within half an ulp."""
    rng = np.random.default_rng(1)
    for _ in range(4000):
        x = float(rng.normal() * 2.0 ** rng.integers(-40, 40))
        e = (math.frexp(x)[1] + 1022) + int(rng.integers(0, 60))
        i = lib.fx_to_fixed(x, e)
        assert abs(i - Fraction(x) * Fraction(2) ** (1079 - e)) <= Fraction(1, 2) and abs(i) <= 1 << 57
        a = int(rng.integers(-(1 << 57), (1 << 57) + 1)) >> int(rng.integers(0, 57))
        sh = int(rng.integers(0, 64))
        assert abs(lib.fx_align(a, sh) - Fraction(a, 1 << sh)) <= Fraction(1, 2)
        assert lib.fx_limbs(a) == a
        v = Fraction(lib.fx_to_double(a, e)) / Fraction(2) ** (e - 1079)
        assert abs(v - a) <= Fraction(abs(a), 1 << 53)
    for a in (0, 1, -1, (1 << 57), -(1 << 57)):
        assert lib.fx_align(a, 0) == a and lib.fx_align(a, 63) == 0 and lib.fx_limbs(a) == a


def _links(rng, kind):
    g = rng.normal(size=(8, 3, 3)) + 1j * rng.normal(size=(8, 3, 3))
    if kind == "unit":
        return np.broadcast_to(np.eye(3, dtype=complex), (8, 3, 3)).copy()
    return np.linalg.qr(g if kind == "random" else np.eye(3) + 1e-3 * g)[0]


def _psi(rng, kind):
    v = rng.normal(size=(8, 4, 3)) + 1j * rng.normal(size=(8, 4, 3))
    if kind == "colours":
        v *= [1.0, 1e-9, 1e-18]
    elif kind == "spins":
        v *= np.array([1e-9, 1.0, 1e-12, 1e-9])[:, None]
    elif kind == "sites":
        v *= 10.0 ** -rng.uniform(0, 12, size=(8, 1, 1))
    elif kind == "components":
        v *= 10.0 ** -rng.uniform(0, 6, size=v.shape)
    elif kind == "one colour":
        v[:, :, 1:] = 0
    elif kind == "point":
        keep = v[3, 1, 2]
        v[:] = 0
        v[3, 1, 2] = keep
    elif kind == "zero spins":
        v[:, 2:] = 0
    elif kind == "large":
        v *= 1e306
    elif kind == "small":
        v *= 1e-300
    return v


def _in_range(v):
    """Whether the exponent word of a block lies in [EX_LOW, EX_HIGH)."""
    return 57 <= max(math.frexp(np.abs(v).max())[1] + 1022, 1) < 2041


KINDS = ["gauss", "colours", "spins", "sites", "components", "one colour", "point", "zero spins", "large", "small"]


@pytest.mark.parametrize("links", ["random", "near unit", "unit"])
@pytest.mark.parametrize("kind", KINDS)
def test_kept_elements_hold_every_component(lib, links, kind):
    rng = np.random.default_rng(10 * KINDS.index(kind) + len(links))
    P = ctypes.POINTER(ctypes.c_double)
    err, units = ctypes.c_double(), ctypes.c_double()
    kept = 0
    for _ in range(1500):
        v = np.ascontiguousarray(_psi(rng, kind)).view(np.float64)
        u = np.ascontiguousarray(_links(rng, links)).view(np.float64)
        keep = lib.fx_element(v.ctypes.data_as(P), u.ctypes.data_as(P), 0, ctypes.byref(err), ctypes.byref(units))
        assert units.value <= 60, (links, kind)
        if kind in ("large", "small"):  # Gaussian fields: kept wherever their exponents are
            assert bool(keep) == _in_range(v)
        if keep:
            kept += 1
            assert err.value <= 61, (links, kind, err.value)
    if kind == "gauss":
        assert kept == 1500  # dense fields are not left to FP64
    if kind == "spins" or (kind == "colours" and links == "unit"):
        assert kept == 0


def test_ends_of_the_exponent_range_are_left_to_fp64(lib):
    P = ctypes.POINTER(ctypes.c_double)
    err, units = ctypes.c_double(), ctypes.c_double()
    rng = np.random.default_rng(5)
    for scale in (1e-285, 1e-295, 1e-308, 3e-310, 1e305, 1.7e308 / 8, 0.0):
        v = np.ascontiguousarray(np.clip(rng.normal(size=(8, 12, 2)), -4, 4) * scale)
        u = np.ascontiguousarray(_links(rng, "random")).view(np.float64)
        assert lib.fx_element(v.ctypes.data_as(P), u.ctypes.data_as(P), 0, ctypes.byref(err), ctypes.byref(units)) == (
            scale == 0.0 or _in_range(v))


@pytest.mark.parametrize("size", [3.0, 0.07, 1.0, 1.41, 1.42, 2.0 ** -60, 1e40])
def test_links_of_other_sizes(lib, size):
    """Rows of norm size: the scale keeps the largest squared norm between 1/2 and 2 (the integer sums then
    stay below 2^63; an overflow would show), and the bounds of unit rows grow by sqrt 2."""
    P = ctypes.POINTER(ctypes.c_double)
    err, units, scale = ctypes.c_double(), ctypes.c_double(), ctypes.c_int()
    assert lib.fx_link_scale(size ** 2, size ** 2, ctypes.byref(scale))
    assert 0.5 <= size ** 2 / 4.0 ** scale.value <= 2
    rng = np.random.default_rng(11)
    for i in range(600):
        v = rng.normal(size=(8, 12, 2))
        if i % 3 == 0:  # the largest sums: every component at the top of its binade
            v = np.sign(v) * (2 - 2.0 ** -52)
        u = np.ascontiguousarray(size * _links(rng, ("random", "near unit", "unit")[i // 200])).view(np.float64)
        v = np.ascontiguousarray(v)
        keep = lib.fx_element(v.ctypes.data_as(P), u.ctypes.data_as(P), scale, ctypes.byref(err), ctypes.byref(units))
        assert units.value <= 60 * 2 ** 0.5
        if keep:
            assert err.value <= 61 * 2 ** 0.5


def test_links_that_do_not_suit(lib):
    s = ctypes.c_int()
    for top, bottom, ok in [(1.0, 1.0, 1), (1.0, 1 / 200, 1), (1.0, 1 / 600, 0), (0.0, 0.0, 0), (float("inf"), 1.0, 0),
                            (float("nan"), 1.0, 0), (1e-300, 1e-300, 0), (1e300, 1e300, 0)]:
        assert lib.fx_link_scale(top, bottom, ctypes.byref(s)) == ok, (top, bottom)
