"""The FP64 collision with per-node coefficients or a reaction source
(fx_collide_general, fx_collide_general3), compiled for the host: each node against
50-digit arithmetic, over flux exponents, C(phi) != phi, both rules for k2, the reaction
term and lattice velocities up to one, and its errors against those of the same
collision in plain FP64."""
import ctypes
import math
import shutil
import subprocess
from decimal import Decimal, getcontext
from fractions import Fraction
from itertools import product
from pathlib import Path

import numpy as np
import pytest

from test_fx import CSRC, TOP, VEL, WGT

NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
getcontext().prec = 50

SRC = r"""
#include "btrt_sweep3.cuh"
using namespace btrt;
namespace {
void halves(double q, int *n, int *h) {   // q = n + h/2, n < 0: neither
    const double t = 2 * q;
    *n = t == floor(t) ? (int)floor(q) : -1;
    *h = t == floor(t) && t != 2 * floor(q);
}
}  // namespace
// c: u^ (dim), bg (dim), q, c3, A0 (upper triangle), a2, k0, k2 (negative: Eq. 62), rate, exponent (rate 0: no
// reaction); many: as many steps per launch compile it; -1: constants refused, 0: node refused
extern "C" int node2(const double *c, double *d, double prev, double *phi, int many) {
    SweepParams<double> p;
    memset(&p, 0, sizeof p);
    p.ux = c[0]; p.uy = c[1]; p.bgx = c[2]; p.bgy = c[3]; p.bq = c[4]; p.bq2 = c[4] == 2.0;
    halves(c[4], &p.bq_n, &p.bq_h);
    p.c3 = c[5]; p.A0xx = c[6]; p.A0xy = c[7]; p.A0yy = c[8]; p.k0 = c[10]; p.k0_one = c[10] == 1.0;
    p.lin.a2x3 = 3 * c[9];
    p.k2_hbb = c[11] < 0; p.k2c = c[11];
    p.react_rate = c[12]; p.react_exp = c[13]; p.react2 = c[13] == 2.0;
    halves(c[13], &p.re_n, &p.re_h);
    p.fx = fx_fold({0, 0, 0}, {0, 0}, {0, 0}, 0, 1 - c[10], {c[0], c[1]}, c[10]);
    p.fx.ok |= (c[2] == c[3] ? kFxSameB : 0) | (c[5] != 0 ? kFxC3 : 0);
    p.fx.trh = 0.5 * (c[6] + c[8]);
    p.fx.detA = c[6] * c[8] - c[7] * c[7];
    if (!(p.fx.ok & kFxOkGeneral)) return -1;
    double (&t)[9] = *reinterpret_cast<double (*)[9]>(d);
    if (many)
        return c[12] != 0 ? fx_collide_general<kGeneral, kSrcReaction, true>(p, t, prev, 0.0, 0, 1.0, *phi)
                          : fx_collide_general<kGeneral, kSrcNone, true>(p, t, prev, 0.0, 0, 0.0, *phi);
    return c[12] != 0 ? fx_collide_general<kGeneral, kSrcReaction>(p, t, prev, 0.0, 0, 1.0, *phi)
                      : fx_collide_general<kGeneral, kSrcNone>(p, t, prev, 0.0, 0, 0.0, *phi);
}
extern "C" int node3(const double *c, double *d, double prev, double *phi) {
    Sweep3Params<double> p;
    memset(&p, 0, sizeof p);
    p.ux = c[0]; p.uy = c[1]; p.uz = c[2]; p.bgx = c[3]; p.bgy = c[4]; p.bgz = c[5]; p.bq = c[6]; p.bq2 = c[6] == 2.0;
    halves(c[6], &p.bq_n, &p.bq_h);
    p.c3 = c[7];
    for (int i = 0; i < 6; ++i) p.A0[i] = c[8 + i];
    p.a2x3 = 3 * c[14]; p.k0 = c[15]; p.k0_one = c[15] == 1.0; p.k2_hbb = c[16] < 0; p.k2c = c[16];
    p.react_rate = c[17]; p.react_exp = c[18]; p.react2 = c[18] == 2.0;
    halves(c[18], &p.re_n, &p.re_h);
    p.src_val = 1.0;
    p.fx = fx_fold3({0, 0, 0, 0, 0, 0}, {0, 0, 0}, {0, 0, 0}, 0, 1 - c[15]);
    if (!(p.fx.ok & kFxOkGeneral)) return -1;
    double (&t)[19] = *reinterpret_cast<double (*)[19]>(d);
    return c[17] != 0 ? fx_collide_general3<kGeneral, kSrcReaction>(p, t, prev, 0.0, *phi)
                      : fx_collide_general3<kGeneral, kSrcNone>(p, t, prev, 0.0, *phi);
}
extern "C" double recip(double v) { return recip_f64(v); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not Path(NVCC).exists():
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("fxg")
    (d / "fx.cu").write_text(SRC)
    subprocess.run([NVCC, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-Xcompiler", "-fPIC,-w,-ffp-contract=off", "-shared", "-I", str(CSRC), str(d / "fx.cu"), "-o",
                    str(d / "fx.so")], check=True, capture_output=True)
    so = ctypes.CDLL(str(d / "fx.so"))
    so.recip.restype = ctypes.c_double
    so.recip.argtypes = [ctypes.c_double]
    return so


def _coeffs(rng, dim, q, c3, k0, k2, rate, umax):
    m, _ = np.linalg.qr(rng.standard_normal((dim, dim)))
    A = (m * rng.uniform(0.005, 0.1, size=dim)) @ m.T
    u = rng.uniform(0.6 * umax, umax, size=dim) * rng.choice([-1.0, 1.0], size=dim)
    bg = rng.uniform(-0.1, 0.1, size=dim)
    if rng.random() < 0.5:
        bg[:] = bg[0]                                       # flux direction (1, 1)
    up = [A[i, j] for i in range(dim) for j in range(i, dim)]
    return [float(t) for t in [*u, *bg, q, c3, *up, rng.uniform(0.0, 0.5), k0, k2, rate, rng.choice([1.0, 1.5, 2.0])]]


def _det(M):
    if len(M) == 2:
        return M[0][0] * M[1][1] - M[0][1] * M[1][0]
    return sum(M[0][i] * (M[1][(i + 1) % 3] * M[2][(i + 2) % 3] - M[1][(i + 2) % 3] * M[2][(i + 1) % 3]) for i in range(3))


def _inverse(M):
    n, det = len(M), _det(M)
    if n == 2:
        return [[M[1][1] / det, -M[0][1] / det], [-M[1][0] / det, M[0][0] / det]]
    return [[(M[(j + 1) % 3][(i + 1) % 3] * M[(j + 2) % 3][(i + 2) % 3]
              - M[(j + 1) % 3][(i + 2) % 3] * M[(j + 2) % 3][(i + 1) % 3]) / det for j in range(3)] for i in range(3)]


def _collide(c, d, prev, num, dim):
    """Eq. 6 with its per-node coefficients in number type `num`; with the result, the sizes of
    what the integer form computes in FP64 (source and C - phi, nonlinear flux, K1 E, k2)."""
    C = VEL[dim]
    c, d, prev = [num(t) for t in c], [num(t) for t in d], num(prev)
    u, bg, q, c3 = c[:dim], c[dim:2 * dim], c[2 * dim], c[2 * dim + 1]
    up = c[2 * dim + 2:-5]
    a2, k0, k2, rate, ex = c[-5:]
    A = [[None] * dim for _ in range(dim)]
    for t, (i, j) in zip(up, [(i, j) for i in range(dim) for j in range(i, dim)]):
        A[i][j] = A[j][i] = t
    power = lambda x, e: x * x if e == 2 else x ** e  # noqa: E731
    phi = sum(d[1:], d[0])
    j = [sum((v[a] * t for v, t in zip(C, d) if v[a]), num(0)) for a in range(dim)]
    s = 3 * (1 + a2 * phi * phi)
    M = [[s * A[a][b] + (num(1) / 2 if a == b else 0) for b in range(dim)] for a in range(dim)]
    K = _inverse(M)
    tr = sum(M[a][a] for a in range(dim))
    if k2 < 0:
        k2 = num(8) * (2 * tr - dim) / (3 * (4 * tr - dim))
    g, gp = power(phi, q), power(prev, q)
    B = [u[a] * phi + bg[a] * g for a in range(dim)]
    dB = [u[a] * (phi - prev) + bg[a] * (g - gp) for a in range(dim)]
    E = [B[a] - dB[a] / 2 - j[a] for a in range(dim)]
    V = [sum(K[a][b] * E[b] for b in range(dim)) + k0 * j[a] + dB[a] for a in range(dim)]
    Cm = c3 * phi * phi * phi
    src = num(0)
    if rate:
        src = (3 * (rate * phi * (1 - power(phi, ex))) - rate * prev * (1 - power(prev, ex))) / 2
    N = {(a, b): sum(v[a] * v[b] * t for v, t in zip(C, d) if v[a] and v[b]) - ((phi + Cm) / 3 if a == b else 0)
         for a in range(dim) for b in range(dim)}
    t3 = sum(N[(a, a)] for a in range(dim)) / 3
    kap = num(9) * (k2 - k0) / 2
    out = []
    for v, w, t in zip(C, WGT[dim], d):
        H = sum(v[a] * v[b] * N[(a, b)] for a in range(dim) for b in range(dim) if v[a] and v[b]) - t3
        w, e2 = num(w.numerator) / num(w.denominator), sum(t * t for t in v)
        z = k0 * (num(3) * e2 / 2 - num(dim) / 2) * Cm
        out.append((1 - k0) * t + w * (k0 * phi + src + z + 3 * sum(v[a] * V[a] for a in range(dim)) - kap * H))
    sizes = (3 * abs(rate) * (abs(phi) + abs(prev)) * 4 + 3 * abs(Cm)
             + 3 * sum(abs(bg[a]) * (abs(g) + abs(gp)) for a in range(dim))
             + 3 * sum(abs(K[a][b]) * abs(E[b]) + abs(K[a][b] * u[b]) * abs(phi) for a in range(dim) for b in range(dim))
             + 5 * (abs(k2) + k0) * sum(abs(n) for n in N.values()))
    return out, phi, sizes


def _node(lib, c, d, prev):
    def run(f, *more):
        t, phi = (ctypes.c_double * len(d))(*d), ctypes.c_double(float("nan"))
        ok = f((ctypes.c_double * len(c))(*c), t, ctypes.c_double(prev), ctypes.byref(phi), *more)
        return ok, list(t), phi.value
    if len(d) != 9:
        return run(lib.node3)
    one, many = run(lib.node2, 0), run(lib.node2, 1)
    assert one[:2] == many[:2] and (one[0] != 1 or one[2] == many[2])   # all kernel forms give the same bits
    return one


def _state(rng, dim):
    phi = rng.uniform(0.3, 1.5)
    return [float(w) * phi * (1 + 0.1 * rng.uniform(-1, 1)) for w in WGT[dim]], phi * (1 + 0.05 * rng.uniform(-1, 1))


FORMS = list(product([2.0, 1.5, 2.3], [0.0, 0.1], [-1.0, 0.7], [0.0, 0.02]))


@pytest.mark.parametrize("dim,umax", [(2, 0.1), (2, 0.45), (2, 0.7), (2, 0.99), (3, 0.1), (3, 0.7)])
@pytest.mark.parametrize("k0", [1.0, 0.83, 1.6])
def test_node_against_exact_arithmetic(lib, dim, k0, umax):
    """The bound of the constant-coefficient form (test_fx.py), and 32 roundings to FP64 of the
    quantities that stay in FP64: K1 by cofactors of a matrix of condition below 4 (16 of
    the 26 operations), powers (pow within 2 ulp), the flux products, the reaction term."""
    rng = np.random.default_rng(int(100 * k0) + int(100 * umax))
    for q, c3, k2, rate in FORMS:
        for _ in range(3):
            c = _coeffs(rng, dim, q, c3, k0, k2, rate, umax)
            d, prev = _state(rng, dim)
            ok, got, phi = _node(lib, c, d, prev)
            assert ok == 1
            ref, rphi, sizes = _collide(c, d, prev, Decimal, dim)
            unit = Decimal(2) ** (math.frexp(max(d))[1] - 1 - TOP[dim])
            ulp = Decimal(2) ** -53
            assert abs(Decimal(phi) - rphi) <= rphi * ulp + 48 * unit
            for g, r in zip(got, ref):
                assert abs(Decimal(g) - r) <= abs(r) * ulp + (48 if dim == 2 else 96) * unit + 32 * ulp * sizes / 9


@pytest.mark.parametrize("k0", [1.0, 1.1])
@pytest.mark.parametrize("dim", [2, 3])
def test_errors_no_larger_than_plain_fp64(lib, dim, k0):
    rng = np.random.default_rng(7)
    e = np.zeros((2, len(VEL[dim]) + 1))
    n = 0
    for _ in range(12):
        for q, c3, k2, rate in FORMS:
            c = _coeffs(rng, dim, q, c3, k0, k2, rate, 0.1)
            d, prev = _state(rng, dim)
            ok, got, phi = _node(lib, c, d, prev)
            assert ok == 1
            ref, rphi, _ = _collide(c, d, prev, Decimal, dim)
            f64, fphi, _ = _collide(c, d, prev, float, dim)
            for k, r in enumerate(ref + [rphi]):
                e[0, k] += float(Decimal((got + [phi])[k]) - r) ** 2
                e[1, k] += float(Decimal((f64 + [fphi])[k]) - r) ** 2
            n += 1
    assert (e[0] <= e[1]).all(), np.sqrt(e / n)


@pytest.mark.parametrize("k0", [1.0, 0.05, 1.4, 1.7, 1.89, 1.98])
@pytest.mark.parametrize("dim", [2, 3])
def test_ends_of_the_word(lib, dim, k0):
    """Populations at the top of a binade, one sign or signs that add up along a direction: right to
    16 roundings of the largest of the sums (20 populations), or refused and untouched."""
    rng = np.random.default_rng(int(100 * k0))
    Q, taken = len(VEL[dim]), 0
    for _ in range(300):
        k2, um, rate = rng.choice([-1.0, 0.02, 0.7, 1.98]), rng.choice([0.05, 0.49, 0.7, 0.99]), rng.choice([0.0, 0.05])
        c = _coeffs(rng, dim, 2.0, rng.choice([0.0, 0.05]), k0, k2, rate, um)
        c[-1] = 2.0
        if rng.random() < 0.3:                              # K1 near 2
            c[2 * dim + 2:-5] = [1e-4 if a == b else 0.0 for a in range(dim) for b in range(a, dim)]
        towards = VEL[dim][rng.integers(0, Q)]
        s = [np.ones(Q), rng.choice([-1.0, 1.0], size=Q), rng.uniform(-1.0, 1.0, size=Q),
             np.array([1.0 if np.dot(towards, v) >= 0 else -1.0 for v in VEL[dim]])][rng.integers(0, 4)]
        top = 0.25 * (2.0 - 2.0 ** -52)
        d, prev = list(rng.choice([-1.0, 1.0]) * top * s), rng.uniform(-4.0, 4.0) * top
        ok, got, phi = _node(lib, c, d, prev)
        taken += ok == 1
        if ok != 1:
            assert got == d
            continue
        ref, rphi, _ = _collide(c, d, prev, Decimal, dim)
        for g, r in zip(got + [phi], ref + [rphi]):
            assert abs(Decimal(g) - r) <= 16 * 20 * Decimal(2) ** -53 * Decimal(top)
    assert taken > 20


@pytest.mark.parametrize("k2", [-1.0, 0.7])
@pytest.mark.parametrize("dim", [2, 3])
def test_coefficients_past_the_reciprocal(lib, dim, k2):
    """Diffusivities so large that the shared reciprocal 1/(det ..) underflows: right or refused."""
    rng = np.random.default_rng(9)
    c = _coeffs(rng, dim, 2.0, 0.0, 1.0, k2, 0.0, 0.1)
    A = [0.05 if a == b else 0.0 for a in range(dim) for b in range(a, dim)]
    c[2 * dim + 2:-5] = A
    d, prev = _state(rng, dim)
    powers = np.arange(230.0, 520.0, 0.25)
    taken = 0
    for e in powers:
        c[-5] = float(2.0 ** e)
        t = list(d)
        ok, got, phi = _node(lib, c, t, prev)
        taken += ok
        if ok != 1:
            assert got == d
            continue
        ref, _, _ = _collide(c, d, prev, Decimal, dim)
        for g, r in zip(got, ref):
            assert abs(Decimal(g) - r) <= Decimal("1e-14")
    assert 0 < taken < len(powers)


def test_reciprocal(lib):
    """Householder's iteration leaves the cube of the seed's error (2^-57 and less) and the rounding
    of its last step."""
    rng = np.random.default_rng(3)
    for v in [1.0, 1.5, 2.0 - 2.0 ** -52, 3.0, 1e-200, 1e200] + list(rng.uniform(1, 2, size=4000)):
        x = Fraction(lib.recip(v)) * Fraction(v)
        assert abs(x - 1) <= Fraction(1, 2 ** 52)
