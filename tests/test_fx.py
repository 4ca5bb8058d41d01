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
// v: K1 - k0 I (xx xy xz yy yz zz), K1 u + g (3), g (3), k2 - k0, k0
extern "C" int node3(const double *v, double *d, double prev, double src, double *phi, int source) {
    FxFold3 q;
    for (int i = 0; i < 6; ++i) q.Q[i] = fx_const(-v[i], 6);
    for (int i = 0; i < 3; ++i) { q.P[i] = fx_const(v[6 + i], 6); q.g[i] = fx_const(-v[9 + i], 6); }
    q.d12 = fx_const(v[12], 12); q.d24 = fx_const(v[12], 24); q.d4 = fx_const(v[12], 4); q.om2 = fx_const(1 - v[13], 2);
    if (!fx_flux_fits3(q.Q[0], q.Q[1], q.Q[2], q.P[0], q.g[0]) || !fx_flux_fits3(q.Q[1], q.Q[3], q.Q[4], q.P[1], q.g[1]) ||
        !fx_flux_fits3(q.Q[2], q.Q[4], q.Q[5], q.P[2], q.g[2])) return -1;
    double (&t)[19] = *reinterpret_cast<double (*)[19]>(d);
    if (v[13] == 1.0)
        return source ? fx_collide_linear3<true, true>(q, t, prev, src, *phi) : fx_collide_linear3<true, false>(q, t, prev, 0, *phi);
    return source ? fx_collide_linear3<false, true>(q, t, prev, src, *phi) : fx_collide_linear3<false, false>(q, t, prev, 0, *phi);
}
extern "C" double convert(long long v, int e, int add) {
    return add ? fx_to_add(v, (unsigned)e << 20) : fx_to(v, (unsigned)e << 20);
}
"""
C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, 1, 0), (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1), (-1, 0, -1),
      (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1)]
VEL = {2: C2, 3: C3}
WGT = {2: [Fraction(4, 9)] + [Fraction(1, 9)] * 4 + [Fraction(1, 36)] * 4,
       3: [Fraction(1, 3)] + [Fraction(1, 18)] * 6 + [Fraction(1, 36)] * 12}
TOP = {2: 58, 3: 57}


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


def _coeffs(rng, k0, dim):
    q, _ = np.linalg.qr(rng.standard_normal((dim, dim)))
    m = 3 * (q * rng.uniform(0.005, 0.4, size=dim)) @ q.T + 0.5 * np.eye(dim)
    K = np.linalg.inv(m)
    u = rng.uniform(-0.1, 0.1, size=dim)
    P = K @ u
    g = u - 0.5 * P
    k1 = dim / np.trace(m)
    pairs = [(i, j) for i in range(dim) for j in range(i, dim)]
    return [float(t) for t in [K[i, j] - (k0 if i == j else 0.0) for i, j in pairs] + list(P + g) + list(g)
            + [8 * (k1 - 2) / (3 * (k1 - 4)) - k0, k0]]


def _collide(v, d, prev, src, num, dim):
    """Eq. 6 in moment form with number type `num` (Fraction: exact; float: rounded at every operation)."""
    C, nq = VEL[dim], dim * (dim + 1) // 2
    v = [num(t) for t in v]
    pairs = [(i, j) for i in range(dim) for j in range(i, dim)]
    Q = dict(zip(pairs, v[:nq]))
    P, g, dk, k0 = v[nq:nq + dim], v[nq + dim:nq + 2 * dim], v[-2], v[-1]
    d, prev, src = [num(t) for t in d], num(prev), num(src)
    phi = sum(d[1:], d[0])
    j = [sum((c[a] * t for c, t in zip(C, d) if c[a]), num(0)) for a in range(dim)]
    V = [P[a] * phi - g[a] * prev - sum(Q[(min(a, b), max(a, b))] * j[b] for b in range(dim)) for a in range(dim)]
    N = {(a, b): sum(c[a] * c[b] * t for c, t in zip(C, d) if c[a] and c[b]) - (phi / 3 if a == b else 0) for a, b in pairs}
    t3 = sum(N[(a, a)] for a in range(dim)) / 3
    a0, kap = k0 * phi + src, num(9) / 2 * dk
    out = []
    for c, w, t in zip(C, WGT[dim], d):
        H = sum((1 if a == b else 2) * c[a] * c[b] * N[(a, b)] for a, b in pairs) - t3
        w = num(w.numerator) / num(w.denominator)
        out.append((1 - k0) * t + w * (a0 + 3 * sum(c[a] * V[a] for a in range(dim)) - kap * H))
    return out, phi


def _node(lib, v, d, prev, src, source):
    t = (ctypes.c_double * len(d))(*d)
    phi = ctypes.c_double(float("nan"))
    f = lib.node if len(d) == 9 else lib.node3
    ok = f((ctypes.c_double * len(v))(*v), t, ctypes.c_double(prev), ctypes.c_double(src), ctypes.byref(phi), source)
    return ok, list(t), phi.value


def _state(rng, kind, dim):
    W, Q = WGT[dim], len(VEL[dim])
    scale = 2.0 ** int(rng.integers(-60, 60))
    if kind == "near":
        d = [float(w) * rng.uniform(0.5, 1.5) * (1 + 0.05 * rng.uniform(-1, 1)) for w in W]
    elif kind == "wide":                   # exponents over the whole word, zeros, signs
        d = [rng.uniform(-1, 1) * 2.0 ** -int(rng.integers(0, 80)) for _ in range(Q)]
        d[int(rng.integers(0, Q))] = 0.0
        d[int(rng.integers(0, Q))] = rng.choice([-1.0, 1.0])
    elif kind == "full":                   # every population at the top of the largest one's binade
        d = [rng.choice([-1.0, 1.0]) * (2.0 - 2.0 ** -52) for _ in range(Q)]
    else:                                  # the ends of the range
        scale = rng.choice([2.0 ** -950, 2.0 ** 1000])
        d = [rng.uniform(-1, 1) for _ in range(Q)]
    d = [t * scale for t in d]
    top = max(abs(t) for t in d)
    return d, float(rng.uniform(-2, 2) * top), float(rng.uniform(-1, 1) * top)


@pytest.mark.parametrize("source", [0, 1])
@pytest.mark.parametrize("k0", [1.0, 0.83, 1.19])
@pytest.mark.parametrize("kind", ["near", "wide", "full", "ends"])
@pytest.mark.parametrize("dim", [2, 3])
def test_node_against_exact_arithmetic(lib, dim, kind, k0, source):
    """Half a unit in the last place of the result, plus units of 2^-58 (three
    dimensions: 2^-57) of the largest population: inputs below the word are cut (one
    each), constants are rounded at 2^-64 and sums once per product; 48 covers their
    weights (96 in three dimensions, with twice the populations)."""
    rng = np.random.default_rng(int(k0 * 100) + source)
    for _ in range(60):
        v = _coeffs(rng, k0, dim)
        d, prev, src = _state(rng, kind, dim)
        ok, got, phi = _node(lib, v, d, prev, src, source)
        assert ok == 1
        ref, rphi = _collide(v, d, prev, src if source else 0.0, Fraction, dim)
        unit = Fraction(2) ** (math.frexp(max(abs(t) for t in d))[1] - 1 - TOP[dim])
        for g, r in zip(got + [phi], ref + [rphi]):
            assert abs(Fraction(g) - r) <= abs(r) * Fraction(1, 2 ** 53) + (48 if dim == 2 else 96) * unit


@pytest.mark.parametrize("k0", [1.0, 1.1])
@pytest.mark.parametrize("dim", [2, 3])
def test_errors_no_larger_than_plain_fp64(lib, dim, k0):
    rng = np.random.default_rng(5)
    e = np.zeros((2, len(VEL[dim]) + 1))
    for _ in range(400):
        v = _coeffs(rng, k0, dim)
        d, prev, src = _state(rng, "near", dim)
        top = Fraction(max(d))
        _, got, phi = _node(lib, v, d, prev, 1e-3 * src, 1)
        ref, rphi = _collide(v, d, prev, 1e-3 * src, Fraction, dim)
        f64, fphi = _collide(v, d, prev, 1e-3 * src, float, dim)
        for k, r in enumerate(ref + [rphi]):
            e[0, k] += float((Fraction((got + [phi])[k]) - r) / top) ** 2
            e[1, k] += float((Fraction((f64 + [fphi])[k]) - r) / top) ** 2
    assert (e[0] <= e[1]).all(), np.sqrt(e / 400)


@pytest.mark.parametrize("dim", [2, 3])
def test_values_out_of_range_are_left_to_fp64(lib, dim):
    v = _coeffs(np.random.default_rng(1), 1.0, dim)
    d = [float(w) for w in WGT[dim]]
    for bad in (float("inf"), float("nan"), 2.0 ** 1019):
        t = d[:3] + [bad] + d[4:]
        ok, got, _ = _node(lib, v, t, 1.0, 0.0, 1)
        assert ok == 0 and got[:3] == t[:3] and got[4:] == t[4:]
        assert _node(lib, v, d, bad, 0.0, 1)[0] == 0
        assert _node(lib, v, d, 1.0, bad, 1)[0] == 0
    ok, got, phi = _node(lib, v, [0.0] * len(d), 0.0, 0.0, 1)
    assert ok == 1 and got == [0.0] * len(d) and phi == 0.0


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
