"""The fixed-point exponential and division of the double-precision solve
(csrc/f64_int.cuh), compiled for the host: against mpmath at 40 digits.  Bounds:
* table: ten roots, each within two units (its own truncation and half its
  predecessor's error), a product of at most ten with half a unit of rounding
  each: below 32 units;
* exponential: a^2 low by at most three units of its last place (2^-56 below
  |a| = 8, 2^-52 above), times ln 2; the polynomial's 32-bit product below 2^-55
  and the table's 32 units of 2^-62: 2^-53.8 below |a| = 8 and 2^-50.8 above,
  plus half an ulp of rounding;
* division: 2^-55 plus half an ulp;
* pivot: operands and products to 2^-59, the reciprocal's square term to 2^-56:
  D within 2^-55 (relative) plus half an ulp, Y within 2^-54.
CPU only."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = """
#include "f64_int.cuh"
static constexpr mgx::Exp2Table tab;
extern "C" double t_exp(uint64_t A) { return mgx::exp2_neg_sq(A, tab.v); }
extern "C" double t_div(double e, double t) { return mgx::div_pos(e, t); }
extern "C" double t_piv(double t, double b, uint64_t *Y) {
    return mgx::from_q62(mgx::pivot_q(mgx::to_q62(t), mgx::to_q62(b) >> 1, *Y));
}
extern "C" void t_pivot(double dt, double dtb, uint64_t *Y, float *D, float *bD) { mgx::pivot(dt, dtb, *Y, *D, *bD); }
extern "C" double t_held(uint64_t Y) { return mgx::held_y(Y); }
extern "C" uint64_t t_hold(double y) { return mgx::hold_y(y); }
extern "C" double t_root(double a) { return mgx::root(a); }
extern "C" uint64_t t_arg(uint64_t alpha, uint64_t g, uint64_t u) { return mgx::arg_magnitude(alpha, g, u); }
extern "C" float t_far(double cc, double ec, double c0, double e0) { return mgx::far_profile(cc, ec, c0, e0); }
extern "C" float t_prod(double b, uint64_t D) { return mgx::narrow_product(b, D); }
extern "C" float t_narrow(uint64_t D) { return mgx::narrow_q62(D); }
extern "C" uint64_t t_tab(int j) { return tab.v[j]; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return compiled(tmp_path_factory, 0)


@pytest.fixture(scope="module", params=[-1, 1])
def moved(request, tmp_path_factory):
    """With the approximate reciprocals as far off as the device's may be."""
    return compiled(tmp_path_factory, request.param)


def compiled(tmp_path_factory, ulps):
    d = tmp_path_factory.mktemp("f64")
    (d / "t.cpp").write_text(SRC)
    so = str(d / "t.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                    f"-DMGX_HOST_ULPS={ulps}", "-I",
                    os.path.join(ROOT, "paper_2011_14998_gb300", "csrc"), str(d / "t.cpp"), "-o", so], check=True)
    L = C.CDLL(so)
    L.t_exp.restype, L.t_exp.argtypes = C.c_double, [C.c_uint64]
    L.t_div.restype, L.t_div.argtypes = C.c_double, [C.c_double, C.c_double]
    L.t_piv.restype, L.t_piv.argtypes = C.c_double, [C.c_double, C.c_double, C.POINTER(C.c_uint64)]
    L.t_pivot.restype, L.t_pivot.argtypes = None, [C.c_double, C.c_double, C.POINTER(C.c_uint64)] + [C.POINTER(C.c_float)] * 2
    L.t_held.restype, L.t_held.argtypes = C.c_double, [C.c_uint64]
    L.t_hold.restype, L.t_hold.argtypes = C.c_uint64, [C.c_double]
    L.t_root.restype, L.t_root.argtypes = C.c_double, [C.c_double]
    L.t_arg.restype, L.t_arg.argtypes = C.c_uint64, [C.c_uint64] * 3
    L.t_far.restype, L.t_far.argtypes = C.c_float, [C.c_double] * 4
    L.t_prod.restype, L.t_prod.argtypes = C.c_float, [C.c_double, C.c_uint64]
    L.t_narrow.restype, L.t_narrow.argtypes = C.c_float, [C.c_uint64]
    L.t_tab.restype, L.t_tab.argtypes = C.c_uint64, [C.c_int]
    return L


def test_table(lib):
    mp.mp.dps = 40
    for j in list(range(0, 1024, 37)) + [1, 511, 512, 1023]:
        assert abs(mp.mpf(lib.t_tab(j)) - mp.mpf(2) ** (62 + mp.mpf(j) / 1024)) < 32


@pytest.mark.parametrize("lo,hi,rel", [(0.0, 1e-3, 2.0 ** -53.8), (0.0, 1.0, 2.0 ** -53.8), (1.0, 8.0, 2.0 ** -53.8),
                                       (8.0, 31.0, 2.0 ** -50.8)])
def test_exponential(lib, lo, hi, rel):
    mp.mp.dps = 40
    rng = np.random.default_rng(int(hi * 10) + int(lo))
    edges = [int(lo * 2 ** 57), int(hi * 2 ** 57) - 1]
    for A in [int(x * 2.0 ** 57) for x in rng.uniform(lo, hi, 4000)] + edges:
        a = mp.mpf(A) / mp.mpf(2) ** 57
        ref = mp.mpf(2) ** (-a * a)
        assert abs(mp.mpf(lib.t_exp(A)) - ref) <= (rel + 2.0 ** -53) * ref
    assert lib.t_exp(0) == 1.0 and lib.t_exp(31 << 57) == 0.0 and lib.t_exp((1 << 64) - 1) == 0.0


def test_division(lib):
    mp.mp.dps = 40
    rng = np.random.default_rng(9)
    e = np.ldexp(rng.uniform(1, 2, 6000), rng.integers(-300, 300, 6000))
    t = np.ldexp(rng.uniform(1, 2, 6000), rng.integers(-300, 300, 6000))
    e[:200] = t[:200] * rng.integers(1, 9, 200)
    t[200:260] = np.ldexp(1.0, rng.integers(-50, 50, 60))
    t[260:320] = np.nextafter(np.ldexp(1.0, rng.integers(-50, 50, 60)), 0.0)
    for x, y in zip(e, t):
        ref = mp.mpf(float(x)) / mp.mpf(float(y))
        assert abs(mp.mpf(lib.t_div(float(x), float(y))) - ref) <= (2.0 ** -55 + 2.0 ** -53) * ref
    # outside the fixed-point range: the plain division
    for x, y in [(0.0, 3.0), (1e-320, 3.0), (3.0, 1e-320), (1e300, 1e-300), (1e-300, 1e300)]:
        with np.errstate(over="ignore", under="ignore"):
            assert lib.t_div(x, y) == float(np.float64(x) / np.float64(y))


def test_pivot(lib):
    """Chains of fixed-point pivots against the recurrence in 40 digits, each step from its own Y."""
    mp.mp.dps = 40
    rng = np.random.default_rng(10)
    for chain in range(60):
        Y, tp = C.c_uint64(1 << 61), 0.0
        for _ in range(60):
            t = float(rng.uniform(0, 1) if chain % 3 == 0 else 10.0 ** rng.uniform(-14, 0))
            b = 0.5 * t + tp
            F = mp.mpf(b) + mp.mpf(Y.value) / mp.mpf(2) ** 61
            D = 1 / (1 + mp.mpf(t) * F)
            got = lib.t_piv(t, b, C.byref(Y))
            assert abs(mp.mpf(got) - D) <= (2.0 ** -55 + 2.0 ** -53) * D
            assert abs(mp.mpf(Y.value) / mp.mpf(2) ** 61 - D * F) <= 2.0 ** -54
            tp = 0.5 * t


def increments(rng, kind, n):
    if kind == "any":
        return 10.0 ** rng.uniform(-12, 6, n)
    if kind == "thick_thin":  # a thick cell, then thin ones
        return np.where(rng.random(n) < 0.3, 10.0 ** rng.uniform(0, 6, n), 10.0 ** rng.uniform(-12, -1, n))
    return np.where(np.arange(n) % 2 == 0, 10.0 ** rng.uniform(-0.1, 0.7), 1e-3)  # around the formats' ends


@pytest.mark.parametrize("kind", ["any", "thick_thin", "ends"])
def test_pivot_of_any_increment(lib, kind):
    """The pivot over chains of increments from 1e-12 to 1e6, Y carried over as between two chunks,
    against the recurrence in 40 digits: D within six roundings of a double and its own to a float;
    Y = D F within eight, or within 2^-53 in fixed point (below 3); over a whole chain the pivot
    F = dtb + Y within eight roundings a row, since dln(D F) / dlnF is at most 1."""
    mp.mp.dps = 40
    rng = np.random.default_rng(14)
    wide = 0
    for _ in range(60):
        Y, tp, ref = C.c_uint64(lib.t_hold(1.0)), 0.0, mp.mpf(1)
        D, bD = C.c_float(), C.c_float()
        for row, t in enumerate(float(x) for x in increments(rng, kind, 60)):
            b = 0.5 * t + tp
            Y.value = lib.t_hold(lib.t_held(Y))  # as put_sweep and get_sweep hand it over
            F = mp.mpf(b) + mp.mpf(lib.t_held(Y))
            d = 1 / (1 + mp.mpf(t) * F)
            lib.t_pivot(t, b, C.byref(Y), C.byref(D), C.byref(bD))
            assert abs(mp.mpf(D.value) - d) <= (6 * 2.0 ** -53 + 2.0 ** -24) * d
            assert abs(mp.mpf(bD.value) - mp.mpf(b) * d) <= (7 * 2.0 ** -53 + 2.0 ** -24 * (1 + 2.0 ** -9)) * mp.mpf(b) * d
            got = mp.mpf(lib.t_held(Y))
            assert abs(got - d * F) <= (8 * 2.0 ** -53) * d * F + (2.0 ** -53 if Y.value < 3 << 61 else 0)
            wide += Y.value >> 63
            ref = 1 / (1 / (mp.mpf(b) + ref) + mp.mpf(t))
            assert abs(got - ref) <= 8 * (row + 1) * 2.0 ** -53 * (0.5 * t + ref)
            tp = 0.5 * t
    assert wide > 100  # the double form was reached


def test_single_precision_results(lib):
    """D and dtb D come out as the nearest floats of the fixed-point D's exact multiples."""
    from fractions import Fraction

    rng = np.random.default_rng(12)
    D = [int(x) for x in rng.integers(1 << 60, 1 << 62, 4000)] + [1 << 62, (1 << 62) - 1, 3 << 60, (1 << 61) + (1 << 37)]
    b = [float(x) for x in 10.0 ** rng.uniform(-40, 0, len(D))]
    for d, x in zip(D, b):
        for got, exact in ((lib.t_narrow(d), Fraction(d, 1 << 62)), (lib.t_prod(x, d), Fraction(x) * Fraction(d, 1 << 62))):
            f = np.float32(got)
            lo, hi = np.nextafter(f, np.float32(0)), np.nextafter(f, np.float32(2))
            err = abs(Fraction(float(f)) - exact)
            # nearest, but for products within 2^-34 of a tie (the high product's error)
            slack = Fraction(float(hi) - float(f)) / (1 << 34)
            assert err <= abs(Fraction(float(lo)) - exact) + slack and err <= abs(Fraction(float(hi)) - exact) + slack


def test_far_lines_leave_the_continuum(lib):
    """From far_profile on a line adds nothing to chi or eta, whatever the values' units (opacities
    and emissivities from 1e-320 to 1e300), and not much nearer it still does."""
    rng = np.random.default_rng(15)
    add = lambda c, x, a: float(Fraction(c) + Fraction(x) * Fraction(2.0 ** -(a * a)))  # fused
    near = 0
    for _ in range(20000):
        cc, ec = (float(10.0 ** rng.uniform(*r)) for r in ((-300, 300), (-320, 300)))
        c0, e0 = float(cc * 10.0 ** rng.uniform(-30, 10)), float(ec * 10.0 ** rng.uniform(-30, 300))
        if rng.random() < 0.2:
            ec = 0.0
        if rng.random() < 0.2:
            c0 = 0.0
        if not (c0 < 1e300 and e0 < 1e300):
            continue
        t = float(np.nextafter(np.float32(lib.t_far(cc, ec, c0, e0)), np.float32(0)))
        if t < 30.9:
            assert add(cc, c0, t) == cc and add(ec, e0, t) == ec
            if t > 1.0:
                near += int(add(cc, c0, t - 0.5) != cc or add(ec, e0, t - 0.5) != ec)
    assert near > 5000
    # an emissivity that is 0 in single precision, beside no continuum emissivity
    assert lib.t_far(1.0, 0.0, 1e-20, 1e-50) == 31.0


def test_profile_argument(lib):
    """|alpha + u gamma| over the whole range the records have, its ends included: exact to three
    units (the product's high half and the shift), or where it passes 31, past 31 as well."""
    rng = np.random.default_rng(16)
    span = [(-63.0, 33.0), (32.5, 33.0), (-63.0, -62.0)]
    for k in range(30000):
        alpha = int(rng.uniform(*span[k % 3]) * 2.0 ** 57)
        gamma = float(rng.uniform(0, 62) if k % 5 else rng.uniform(61, 62)) if k % 2 else float(10.0 ** rng.uniform(-6, 0))
        sh = max(0, min(4, 5 - (int(np.frexp(gamma / 2)[1]))))
        g = int(gamma * 2.0 ** 57) << sh & ~7 | sh
        u = int(rng.integers(0, 1 << 63)) if k % 7 else (1 << 63) - 1
        assert g < 1 << 63
        got = lib.t_arg(alpha & ((1 << 64) - 1), g, u)
        exact = abs(alpha + (u * (g & ~7) >> 63 >> sh))
        if exact >= 31 << 57:
            assert got >= 31 << 57
        else:
            assert abs(got - exact) <= 3


def test_division_and_pivot_with_other_reciprocals(moved):
    test_division(moved)
    test_pivot(moved)
    test_pivot_of_any_increment(moved, "thick_thin")


def check_root(L):
    mp.mp.dps = 40
    rng = np.random.default_rng(17)
    a = np.concatenate([10.0 ** rng.uniform(-36, 36, 6000), rng.uniform(1, 4, 2000), np.arange(1, 200.0) ** 2])
    for x in a:
        ref = mp.sqrt(mp.mpf(float(x)))
        ulp = mp.mpf(2) ** (int(mp.floor(mp.log(ref, 2))) - 52)
        # two corrections leave 2^-64 before the last rounding
        assert abs(mp.mpf(L.t_root(float(x))) - ref) <= (0.5 + 2.0 ** -10) * ulp
    for x in (0.0, 1e-300, 5e-324, 1e300):
        assert L.t_root(x) == np.sqrt(x)


def test_root(lib):
    check_root(lib)


def test_root_with_other_reciprocals(moved):
    check_root(moved)
