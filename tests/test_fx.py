"""The FP64 collision's integer form (csrc/btrt_fx.cuh), compiled for the host: each
node against exact rational arithmetic, and its errors against those of the same
collision in plain FP64."""
import ctypes
import math
import shutil
import subprocess
from fractions import Fraction
from pathlib import Path

import numpy as np
import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_1902_09813_gb300" / "csrc"
SRC = r"""
#include "btrt_fx.cuh"
using namespace btrt;
// v: Qxx Qxy Qyy Px Py gx gy (K1 - k0 I, K1 u + g, g), k2 - k0, k0
extern "C" int node(const double *v, double *d, double prev, double src, double *phi, int source) {
    FxFold q;
    q.Qxx = fx_const(-v[0], 6); q.Qxy = fx_const(-v[1], 6); q.Qyy = fx_const(-v[2], 6);
    q.Px = fx_const(v[3], 6); q.Py = fx_const(v[4], 6); q.gx = fx_const(-v[5], 6); q.gy = fx_const(-v[6], 6);
    q.d18 = fx_const(v[7], 18); q.d4 = fx_const(v[7], 4); q.om2 = fx_const(1 - v[8], 2);
    if (!fx_flux_fits(q.Qxx, q.Qxy, q.Px, q.gx) || !fx_flux_fits(q.Qxy, q.Qyy, q.Py, q.gy)) return -1;
    double (&t)[9] = *reinterpret_cast<double (*)[9]>(d);
    if (v[8] == 1.0)
        return source ? fx_collide_linear<true, true>(q, t, prev, src, *phi) : fx_collide_linear<true, false>(q, t, prev, 0, *phi);
    return source ? fx_collide_linear<false, true>(q, t, prev, src, *phi) : fx_collide_linear<false, false>(q, t, prev, 0, *phi);
}
extern "C" double convert(long long v, int e, int add) {
    return add ? fx_to_add(v, (unsigned)e << 20) : fx_to(v, (unsigned)e << 20);
}
"""
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = [Fraction(4, 9)] + [Fraction(1, 9)] * 4 + [Fraction(1, 36)] * 4


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-I", str(CSRC), str(d / "fx.cpp"), "-o",
                    str(d / "fx.so")], check=True)
    so = ctypes.CDLL(str(d / "fx.so"))
    so.convert.restype = ctypes.c_double
    so.convert.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int]
    return so


def _coeffs(rng, k0):
    l1, l2, th = rng.uniform(0.005, 0.4), rng.uniform(0.005, 0.4), rng.uniform(0, math.pi)
    c, s = math.cos(th), math.sin(th)
    xx, yy, xy = 3 * (l1 * c * c + l2 * s * s) + 0.5, 3 * (l1 * s * s + l2 * c * c) + 0.5, 3 * (l1 - l2) * c * s
    det = xx * yy - xy * xy
    K = (yy / det, -xy / det, xx / det)
    u = rng.uniform(-0.1, 0.1, size=2)
    P = (K[0] * u[0] + K[1] * u[1], K[1] * u[0] + K[2] * u[1])
    g = (u[0] - 0.5 * P[0], u[1] - 0.5 * P[1])
    k1 = 2 / (xx + yy)
    return [K[0] - k0, K[1], K[2] - k0, P[0] + g[0], P[1] + g[1], g[0], g[1], 8 * (k1 - 2) / (3 * (k1 - 4)) - k0, k0]


def _collide(v, d, prev, src, num):
    """Eq. 6 in moment form with number type `num` (Fraction: exact; float: rounded at every operation)."""
    Qxx, Qxy, Qyy, Px, Py, gx, gy, dk, k0 = (num(t) for t in v)
    d, prev, src = [num(t) for t in d], num(prev), num(src)
    phi = sum(d[1:], d[0])
    jx, jy = (sum((e * t for e, t in zip(E, d) if e), num(0)) for E in (EX, EY))
    V = (Px * phi - gx * prev - Qxx * jx - Qxy * jy, Py * phi - gy * prev - Qxy * jx - Qyy * jy)
    nxx = sum(d[i] for i in range(9) if EX[i]) - phi / 3
    nyy = sum(d[i] for i in range(9) if EY[i]) - phi / 3
    nxy = d[5] + d[7] - d[6] - d[8]
    a, kap = k0 * phi + src, num(9) / 2 * dk
    out = []
    for i in range(9):
        H = (EX[i] ** 2) * nxx + (EY[i] ** 2) * nyy + 2 * EX[i] * EY[i] * nxy - (nxx + nyy) / 3
        w = num(W[i].numerator) / num(W[i].denominator)
        out.append((1 - k0) * d[i] + w * (a + 3 * (EX[i] * V[0] + EY[i] * V[1]) - kap * H))
    return out, phi


def _node(lib, v, d, prev, src, source):
    t = (ctypes.c_double * 9)(*d)
    phi = ctypes.c_double(float("nan"))
    ok = lib.node((ctypes.c_double * 9)(*v), t, ctypes.c_double(prev), ctypes.c_double(src), ctypes.byref(phi), source)
    return ok, list(t), phi.value


def _state(rng, kind):
    scale = 2.0 ** int(rng.integers(-60, 60))
    if kind == "near":
        d = [float(w) * rng.uniform(0.5, 1.5) * (1 + 0.05 * rng.uniform(-1, 1)) for w in W]
    elif kind == "wide":                   # exponents over the whole word, zeros, signs
        d = [rng.uniform(-1, 1) * 2.0 ** -int(rng.integers(0, 80)) for _ in range(9)]
        d[int(rng.integers(0, 9))] = 0.0
        d[int(rng.integers(0, 9))] = rng.choice([-1.0, 1.0])
    elif kind == "full":                   # every population at the top of the largest one's binade
        d = [rng.choice([-1.0, 1.0]) * (2.0 - 2.0 ** -52) for _ in range(9)]
    else:                                  # the ends of the range
        scale = rng.choice([2.0 ** -950, 2.0 ** 1000])
        d = [rng.uniform(-1, 1) for _ in range(9)]
    d = [t * scale for t in d]
    top = max(abs(t) for t in d)
    return d, float(rng.uniform(-2, 2) * top), float(rng.uniform(-1, 1) * top)


@pytest.mark.parametrize("source", [0, 1])
@pytest.mark.parametrize("k0", [1.0, 0.83, 1.19])
@pytest.mark.parametrize("kind", ["near", "wide", "full", "ends"])
def test_node_against_exact_arithmetic(lib, kind, k0, source):
    """Half a unit in the last place of the result, plus units of 2^-58 of the largest
    population: inputs below the word are cut (one each, nine of them), constants are
    rounded at 2^-64 and sums once per product; 48 covers their weights."""
    rng = np.random.default_rng(int(k0 * 100) + source)
    for _ in range(60):
        v = _coeffs(rng, k0)
        d, prev, src = _state(rng, kind)
        ok, got, phi = _node(lib, v, d, prev, src, source)
        assert ok == 1
        ref, rphi = _collide(v, d, prev, src if source else 0.0, Fraction)
        unit = Fraction(2) ** (math.frexp(max(abs(t) for t in d))[1] - 1 - 58)
        for g, r in zip(got + [phi], ref + [rphi]):
            assert abs(Fraction(g) - r) <= abs(r) * Fraction(1, 2 ** 53) + 48 * unit


@pytest.mark.parametrize("k0", [1.0, 1.1])
def test_errors_no_larger_than_plain_fp64(lib, k0):
    rng = np.random.default_rng(5)
    e = np.zeros((2, 10))
    for _ in range(400):
        v = _coeffs(rng, k0)
        d, prev, src = _state(rng, "near")
        top = Fraction(max(d))
        _, got, phi = _node(lib, v, d, prev, 1e-3 * src, 1)
        ref, rphi = _collide(v, d, prev, 1e-3 * src, Fraction)
        f64, fphi = _collide(v, d, prev, 1e-3 * src, float)
        for k, r in enumerate(ref + [rphi]):
            e[0, k] += float((Fraction((got + [phi])[k]) - r) / top) ** 2
            e[1, k] += float((Fraction((f64 + [fphi])[k]) - r) / top) ** 2
    assert (e[0] <= e[1]).all(), np.sqrt(e / 400)


def test_values_out_of_range_are_left_to_fp64(lib):
    v = _coeffs(np.random.default_rng(1), 1.0)
    d = [float(w) for w in W]
    for bad in (float("inf"), float("nan"), 2.0 ** 1019):
        t = d[:3] + [bad] + d[4:]
        ok, got, _ = _node(lib, v, t, 1.0, 0.0, 1)
        assert ok == 0 and got[:3] == t[:3] and got[4:] == t[4:]
        assert _node(lib, v, d, bad, 0.0, 1)[0] == 0
        assert _node(lib, v, d, 1.0, bad, 1)[0] == 0
    ok, got, phi = _node(lib, v, [0.0] * 9, 0.0, 0.0, 1)
    assert ok == 1 and got == [0.0] * 9 and phi == 0.0


def test_conversions(lib):
    rng = np.random.default_rng(2)
    values = [0, 1, -1, 2 ** 53 - 1, 2 ** 53 + 1, 2 ** 54 + 3, -(2 ** 54) - 2, 2 ** 62 - 1, -(2 ** 62) + 1, 2 ** 32, 2 ** 32 - 1]
    values += [int(rng.integers(-2 ** 62, 2 ** 62)) >> int(rng.integers(0, 62)) for _ in range(2000)]
    for x in values:
        for e in (64, 1023, 2040):
            want = Fraction(x) * Fraction(2) ** (e - 1023 - 58)
            for add in (0, 1):
                got = Fraction(lib.convert(x, e, add))
                assert abs(got - want) <= abs(want) * Fraction(1, 2 ** 53)
