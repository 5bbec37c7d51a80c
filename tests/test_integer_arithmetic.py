"""The kernels' integer arithmetic, built for the host, against exact rational numbers.

eri_scalar.cuh (scalars of a primitive quartet), rys_fixed.h (root polynomials) and eri_fixed.cuh
(the fixed-point sums of Eq. 1) compile on the host; the bounds below are those that
their operations have: the units that each rounding or dropped product may be off by."""

import ctypes
import os
import random
import shutil
import subprocess
from fractions import Fraction as Fr
from math import frexp, isqrt

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2407_09700_gb300", "csrc")
I64, D, INT = ctypes.c_int64, ctypes.c_double, ctypes.c_int


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    so = str(tmp_path_factory.mktemp("host") / "host_fixed_point.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, os.path.join(HERE, "host_fixed_point.cpp"),
                    os.path.join(CSRC, "rys_table.cpp"), "-o", so], check=True)
    h = ctypes.CDLL(so)
    h.host_rsqrt.restype = h.host_horner.restype = I64
    h.host_rsqrt.argtypes = [I64]
    h.host_sum.restype = D
    return h


def test_reciprocal_square_root(lib):
    # y within 8 units of 2^-60: four truncated or rounded products, and 5/16 e^3 below 2^-61
    rng = random.Random(1)
    fs = [1 << 60, (1 << 62) - 1, (1 << 61) - 1, 1 << 61] + [int(2 ** rng.uniform(60, 62)) for _ in range(20000)]
    for f in fs:
        assert abs(lib.host_rsqrt(f) - isqrt((1 << 180) // f)) <= 8


def test_places_of_a_sides_unit(lib):
    # p places leave c (units of 2^-60) and f 2^(e - 62) below a half, one more leaves one of them at a
    # half or above
    rng = random.Random(3)
    for t in range(4000):
        c = [rng.choice((-1, 1)) * int(2 ** rng.uniform(0, 60)) if rng.random() < 0.7 else 0 for _ in range(3)]
        f, e = int(2 ** rng.uniform(0, 62)), rng.randrange(-70, 1)
        p = lib.host_places1((I64 * 3)(*c), I64(f), INT(e))
        big = max([Fr(abs(x), 1 << 60) for x in c] + [Fr(f) * Fr(2) ** (e - 62)])
        # a negative c counts as one more than its size does: exact powers of two
        assert p >= 0 and (p == 0 or big * 2 ** p <= Fr(1, 2))
        assert big * 2 ** (p + 1) >= Fr(1, 2) or p == 59


def test_scalars_of_a_primitive_quartet(lib):
    rng = random.Random(2)
    tcut = 41
    out = (I64 * 14)()
    seen = set()
    for t in range(4000):
        pu = rng.randrange(30, 59)
        ze = [10.0 ** rng.uniform(-3, 10) for _ in range(2)]
        if t % 5 == 0:
            ze[1] = ze[0]
        P = [rng.randrange(-(1 << 58), 1 << 58) for _ in range(3)]
        sep = 10.0 ** rng.uniform(-3, 4) / max(min(ze), 1e-3) ** 0.5
        Q = [p - max(-(1 << 59), min(1 << 59, int(sep * rng.uniform(-1, 1) * 2.0 ** pu))) for p in P]
        if t % 50 == 0:
            Q = list(P)
        H = 1 / ze[0] + 1 / ze[1]
        lib.host_quartet(D(H), (I64 * 3)(*P), (I64 * 3)(*Q), INT(pu), I64(4 * tcut << 54), out)
        g, ge, d0, d1, d2, k, ti, x0, x1, rT, rTe, rT2, g2, g2e = out
        H = Fr(H)
        for d, p, q in zip((d0, d1, d2), P, Q):         # P - Q is exact
            assert Fr(d) * Fr(2) ** (k - 60) == Fr(p - q) / 2 ** pu and abs(d) <= 1 << 60
        gg = Fr(g2) * Fr(2) ** (g2e - 62)               # rho: twice g's 8 units of 2^-60, and its product's
        assert abs(gg * H - 1) <= Fr(20, 1 << 60)
        T = sum(Fr(p - q) ** 2 for p, q in zip(P, Q)) / 4 ** pu / H
        if ti >= 0:
            # rho's error and the lookup's 2^-56; next to an interval's end its neighbour may serve
            x = (Fr((x0 << 29) + x1) / (1 << 60) + 1) / 2
            assert abs((ti + x) / 4 - T) <= T * Fr(40, 1 << 60) + Fr(4, 1 << 56)
            assert T < tcut + Fr(1, 1 << 40) and 0 <= x <= 1
            seen.add("near")
        else:
            assert T > tcut - Fr(1, 1 << 40)
            r = Fr(rT) * Fr(2) ** (rTe - 62)
            assert abs(r * r * T - 1) <= Fr(60, 1 << 60)
            assert abs(Fr(rT2) * Fr(2) ** (2 * rTe - 62) * T - 1) <= Fr(60, 1 << 60)
            assert Fr(1, 2) ** 2 * Fr(2) ** (2 * rTe) <= 1 / T * Fr(1001, 1000)    # the weights' unit: within 2 of 1 / sqrt(T)
            seen.add("far")
    assert seen == {"near", "far"}


def _table(lib, N):
    deg, sub, tcut, off, coef = INT(), INT(), INT(), ctypes.c_longlong(), ctypes.POINTER(D)()
    lib.host_table(N, *(ctypes.byref(v) for v in (deg, sub, tcut, off, coef)))
    return deg.value, sub.value, tcut.value, off.value, coef


@pytest.mark.parametrize("N", [1, 2, 3, 5, 9])
def test_root_polynomials(lib, N):
    rng = random.Random(N)
    deg, sub, tcut, off, coef = _table(lib, N)
    for _ in range(300):
        i = rng.randrange(0, sub * tcut)
        T = (i + rng.random()) / sub
        for r in range(2 * N):                          # u and w of every root
            o = off + (i * N * 2 + r) * (deg + 1)
            c = (D * (deg + 1))(*coef[o:o + deg + 1])
            E, ti, x60 = INT(), INT(), I64()
            v = lib.host_horner(c, D(T), ctypes.byref(E), ctypes.byref(ti), ctypes.byref(x60))
            assert ti.value == int(sub * T)
            x = Fr(x60.value, 1 << 60)
            assert abs(x - (2 * (sub * Fr(T) - ti.value) - 1)) <= Fr(1, 1 << 54)
            want = Fr(0)
            for k in range(deg + 1):
                want = want * x + Fr(c[k])
            # units of 2^(E - 62): half a one for each of seven coefficients and 32 for the short one, and five a
            # step: three bits of the sum and the product of the low halves, and one for the shift
            assert abs(v * Fr(2) ** (E.value - 62) - want) <= 72 * Fr(2) ** (E.value - 62)


def _biased(v):
    return frexp(v)[1] + 1022 if v else 0


# Each factor's error is half a unit of its limbs (2^-57 of its scale for x, 2^-58 for y and z), the
# product's one unit of 2^-57 and each sum's dropped limb products two of 2^-60 or so: 32 terms within
# 32 * 4 * 2^-57 of the product of the three scales.  With one exponent per factor, that product is
# below eight times the largest term's.
@pytest.mark.parametrize("spread", [0, 3, 25])
def test_fixed_point_sums(lib, spread):
    rng = random.Random(spread)
    for n in [1, 2, 3, 7, 31, 32] * 50:
        v = [[rng.choice((-1, 1)) * rng.uniform(0.5, 1.0) * 2.0 ** (c + rng.randint(-spread, 0)) for _ in range(n)]
             for c in (17, -5, 100)]
        if n > 2:
            v[0][1] = 0.0
            v[1][2] = 5e-324                            # a denormal counts as zero
        K = [max(_biased(x) for x in w) for w in v]
        got = lib.host_sum(INT(n), *((D * n)(*w) for w in v), (INT * 3)(*K))
        want = sum(Fr(a) * Fr(b) * Fr(c) for a, b, c in zip(*v))
        scale = Fr(2) ** (sum(K) - 3 * 1022)
        assert abs(Fr(got) - want) <= 4 * n * scale / 2 ** 57 + abs(want) / 2 ** 53

