"""Range of the FP64 collision's integer form (csrc/btrt_fx.cuh): states that take its
sums to the ends of the 64-bit word must come out right or be left to the FP64 form,
for every relaxation parameter a lattice takes."""
import ctypes
import math
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from test_fx import CSRC, TOP, VEL, WGT, _coeffs, _collide, _state

SRC = r"""
#include "btrt_fx.cuh"
using namespace btrt;
// v: K1 - k0 I, K1 u + g, g, k2 - k0, k0 (as in test_fx.py); -1: constants refused, 0: node refused
extern "C" int node2(const double *v, double *d, double prev, double src, double *phi, int source) {
    const FxFold q = fx_fold({v[0], v[1], v[2]}, {v[3], v[4]}, {v[5], v[6]}, v[7], 1 - v[8], {0, 0}, v[8]);
    if (!(q.ok & kFxOkLinear)) return -1;
    double (&t)[9] = *reinterpret_cast<double (*)[9]>(d);
    if (v[8] == 1.0)
        return source ? fx_collide_linear<true, true>(q, t, prev, src, *phi) : fx_collide_linear<true, false>(q, t, prev, 0, *phi);
    return source ? fx_collide_linear<false, true>(q, t, prev, src, *phi) : fx_collide_linear<false, false>(q, t, prev, 0, *phi);
}
extern "C" int node3(const double *v, double *d, double prev, double src, double *phi, int source) {
    const FxFold3 q = fx_fold3({v[0], v[1], v[2], v[3], v[4], v[5]}, {v[6], v[7], v[8]}, {v[9], v[10], v[11]}, v[12], 1 - v[13]);
    if (!(q.ok & kFxOkLinear)) return -1;
    double (&t)[19] = *reinterpret_cast<double (*)[19]>(d);
    if (v[13] == 1.0)
        return source ? fx_collide_linear3<true, true>(q, t, prev, src, *phi) : fx_collide_linear3<true, false>(q, t, prev, 0, *phi);
    return source ? fx_collide_linear3<false, true>(q, t, prev, src, *phi) : fx_collide_linear3<false, false>(q, t, prev, 0, *phi);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fxr")
    (d / "fx.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-I", str(CSRC), str(d / "fx.cpp"), "-o",
                    str(d / "fx.so")], check=True)
    return ctypes.CDLL(str(d / "fx.so"))


def _node(lib, v, d, prev, src, source):
    t = (ctypes.c_double * len(d))(*d)
    phi = ctypes.c_double(float("nan"))
    f = lib.node2 if len(d) == 9 else lib.node3
    ok = f((ctypes.c_double * len(v))(*v), t, ctypes.c_double(prev), ctypes.c_double(src), ctypes.byref(phi), source)
    return ok, list(t), phi.value


def _srt(k0, k2, dim):
    """K1 = k0 I, no flux: the constants of a single relaxation rate (k2 = k0) and beyond."""
    return [0.0] * (dim * (dim + 1) // 2 + 2 * dim) + [k2 - k0, k0]


def _top_states(rng, v, dim):
    """Every population at the top of its binade, with the signs that drive one result or
    all of phi to its largest size; phi^{n-1} and the source as large as the form admits."""
    Q = len(VEL[dim])
    top, prev, src = 2.0 - 2.0 ** -52, 8.0 - 2.0 ** -50, 4.0 - 2.0 ** -51
    yield [top] * Q, top, 0.0
    yield [top] * Q, prev, src
    yield [-top] * Q, -prev, -src
    yield [top - rng.uniform(0, 0.4) for _ in range(Q)], prev, src
    unit = np.eye(Q)
    rows = np.array([_collide(v, list(unit[k]), 0.0, 0.0, float, dim)[0] for k in range(Q)])
    of_prev = _collide(v, [0.0] * Q, 1.0, 0.0, float, dim)[0]
    for i in range(Q):
        s = np.where(rows[:, i] < 0, -1.0, 1.0)
        yield list(s * top), math.copysign(prev, of_prev[i]), src


@pytest.mark.parametrize("source", [0, 1])
@pytest.mark.parametrize("k0", [0.001, 0.1, 1.0, 1.3, 1.5, 1.6, 1.7, 1.8, 1.9, 1.99, 1.9997])
@pytest.mark.parametrize("dim", [2, 3])
def test_ends_of_the_word(lib, dim, k0, source):
    """Right (the bound of test_fx.py's exact comparison) or refused with the populations untouched."""
    rng = np.random.default_rng(int(1000 * k0))
    consts = [_srt(k0, k2, dim) for k2 in (k0, 0.001, 0.5, 1.999)] + [_coeffs(rng, k0, dim) for _ in range(6)]
    for v in consts:
        for d, prev, src in _top_states(rng, v, dim):
            ok, got, phi = _node(lib, v, d, prev, src, source)
            if ok != 1:
                assert got == d
                continue
            ref, rphi = _collide(v, d, prev, src if source else 0.0, Fraction, dim)
            unit = Fraction(2) ** (math.frexp(max(abs(t) for t in d))[1] - 1 - TOP[dim])
            for g, r in zip(got + [phi], ref + [rphi]):
                assert abs(Fraction(g) - r) <= abs(r) * Fraction(1, 2 ** 53) + (48 if dim == 2 else 96) * unit


@pytest.mark.parametrize("dim", [2, 3])
def test_ordinary_states_are_not_refused(lib, dim):
    rng = np.random.default_rng(4)
    for k0 in (0.01, 0.3, 1.0, 1.6, 1.9, 1.99):
        for _ in range(40):
            v = _coeffs(rng, k0, dim)
            d, prev, src = _state(rng, "near", dim)
            assert _node(lib, v, d, prev, 0.1 * src, 1)[0] == 1
            full = [float(w) * (1 + 0.1 * rng.uniform(-1, 1)) for w in WGT[dim]]
            assert _node(lib, v, full, 1.0, 0.1, 1)[0] == 1


@pytest.mark.parametrize("k0", [1.0, 1.1])
@pytest.mark.parametrize("dim", [2, 3])
def test_tiny_nodes_are_left_to_fp64(lib, dim, k0):
    """Below 2^-959 the integers' unit would be coarser than FP64's own: such nodes are refused
    with the populations untouched; a node of zeros is not."""
    v = _coeffs(np.random.default_rng(1), k0, dim)
    Q = len(VEL[dim])
    for e in (-965, -1000, -1030, -1070):
        d = [float(t) * 2.0 ** e for t in WGT[dim]]
        ok, got, _ = _node(lib, v, d, 2.0 ** e, 0.0, 0)
        assert ok == 0 and got == d
        for k in range(Q):
            one = [0.0] * Q
            one[k] = -(2.0 ** e)
            ok, got, _ = _node(lib, v, one, 0.0, 0.0, 0)
            assert ok == 0 and got == one
        assert _node(lib, v, [0.0] * Q, 2.0 ** e, 0.0, 1)[0] == 0
        assert _node(lib, v, [0.0] * Q, 0.0, -(2.0 ** e), 1)[0] == 0
    for z in (0.0, -0.0):
        ok, got, phi = _node(lib, v, [z] * Q, z, z, 1)
        assert ok == 1 and got == [0.0] * Q and phi == 0.0
    d = [float(t) * 2.0 ** -955 for t in WGT[dim]]
    assert _node(lib, v, d, 2.0 ** -955, 0.0, 0)[0] == 1
