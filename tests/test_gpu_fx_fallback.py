"""FP64 lattices whose nodes or constants the integer collision does not take
(csrc/btrt_fx.cuh): the out-of-line FP64 forms on the device, beside nodes that stay on
the integer form, against the FP64 oracle."""
import ctypes
from fractions import Fraction

import numpy as np
import pytest

import oracle
import workloads as w
from conftest import cpu_threads
from oracle import d3q19 as o3

pytestmark = pytest.mark.gpu

TOL64 = 1e-11
COEFFS = {"linear": dict(), "general": dict(b2=0.05, c3=0.02, a2=0.3), "reaction": dict()}


def _rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def _problem(dim, kind, bc=0, seed=3, source="const"):
    if dim == 2:
        p = w.random_state_problem(45, 38, seed=seed, bc=(0, 0, bc, bc), nonlinear=False, source=source)
    else:
        p = w.random_state_problem3(13, 11, 10, seed=seed, bc=(0, 0, bc, bc, 0, 0), nonlinear=False, source=source)
    p = p.replace(**COEFFS[kind])
    if kind == "reaction":
        p.source.kind, p.source.const, p.source.exp = "reaction", 0.02, 1.5
    return p


def _run(p, field, steps):
    """GPU and oracle after `steps`: phi and the populations the GPU keeps then."""
    from paper_1902_09813_gb300 import Lattice, Lattice3
    if field.ndim == 2:
        ref = oracle.OracleLattice(p.replace(phi0_array=field), nthreads=cpu_threads()).init()
        lat = Lattice.from_problem(p, compute="f64")
    else:
        ref = o3.OracleLattice3(p.replace(phi0_fn=lambda X, Y, Z: field), nthreads=cpu_threads()).init()
        lat = Lattice3.from_problem(p, compute="f64")
    lat.init(field).step(steps)
    ref.step(steps)
    phi = ref.phi()
    ref.step(1)
    assert lat.check() == 0
    return lat.phi_host(), phi, lat.read_f(), ref.fpost.copy()


@pytest.mark.parametrize("steps", [1, 3])
@pytest.mark.parametrize("kind", COEFFS)
@pytest.mark.parametrize("dim", [2, 3])
def test_constants_that_do_not_fit(dim, kind, steps):
    """k0 = 1e-4 clears both forms' bits (1 - k0 does not fit)."""
    p = _problem(dim, kind, bc=1).replace(k0=1e-4)
    got, phi, f, fpost = _run(p, p.phi0(), steps)
    assert _rel(got, phi) <= TOL64 and _rel(f, fpost) <= TOL64


@pytest.mark.parametrize("kind", ["linear", "general"])
@pytest.mark.parametrize("dim", [2, 3])
def test_velocities_that_do_not_fit(dim, kind):
    p = _problem(dim, kind).replace(u=(2.4, -2.2, 2.0)[:dim])
    got, phi, f, fpost = _run(p, p.phi0(), 2)
    assert _rel(got, phi) <= TOL64 and _rel(f, fpost) <= TOL64


def _local_max(a, steps):
    """Largest magnitude that reaches a node within `steps` steps."""
    m = np.abs(a)
    for _ in range(steps + 1):
        for ax in range(a.ndim):
            m = np.maximum(m, np.maximum(np.roll(m, 1, axis=ax), np.roll(m, -1, axis=ax)))
    return m


@pytest.mark.parametrize("steps", [1, 4])
@pytest.mark.parametrize("kind", COEFFS)
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("k0", [1.0, 1.15])
def test_rough_fields(dim, kind, steps, k0):
    """Log-normal fields over eight decades: phi^{n-1}, the source or the flux of many nodes lie out
    of reach of their populations; errors are measured against what surrounds a node."""
    p = _problem(dim, kind, bc=1).replace(k0=k0)
    field = np.exp(np.random.default_rng(8).normal(-6.0, 3.0, size=p.phi0().shape))
    got, phi, f, fpost = _run(p, field, steps)
    assert _rel(got, phi) <= TOL64 and _rel(f, fpost) <= TOL64
    if dim == 2 and kind == "linear":
        near = _local_max(field, steps) + abs(p.source.const)
        inner = slice(steps + 2, -steps - 2)                         # off the walls' values
        assert np.all(np.abs(got - phi)[inner] <= TOL64 * near[inner])


@pytest.mark.parametrize("k0", [1.0, 1.2])
@pytest.mark.parametrize("dim", [2, 3])
def test_values_above_the_range(dim, k0):
    """A source that lifts part of a field past the largest exponent the integers take, 2^1017, step
    by step, against the same linear problem 2^900 times smaller (the oracle squares phi)."""
    from paper_1902_09813_gb300 import Lattice, Lattice3
    out = []
    for scale in (1.0, 2.0 ** -900):
        p = _problem(dim, "linear", source="const").replace(k0=k0)
        p.source.const = (2.5e305 if dim == 2 else 4.5e305) * scale
        field = scale * (1.2e306 + 8e305 * p.phi0() / np.max(p.phi0()))
        lat = (Lattice if dim == 2 else Lattice3).from_problem(p, compute="f64").init(field).step(6)
        assert lat.check() == 0
        out.append((lat.phi_host() * (2.0 ** -1000 / scale), lat.read_f() * (2.0 ** -1000 / scale)))
    (phi_a, f_a), (phi_b, f_b) = out
    largest = np.max(np.abs(f_a), axis=0)
    assert np.any(largest > 2.0 ** 17)                               # the initial field's lie below
    assert _rel(phi_a, phi_b) <= TOL64 and _rel(f_a, f_b) <= TOL64


def test_reciprocal():
    """The sweeps' reciprocal over mantissas and exponents: half a unit in the last place and the rest
    of Householder's iteration, 2^-52 of the result in all."""
    import torch
    from paper_1902_09813_gb300 import _capi as C
    rng = np.random.default_rng(2)
    v = np.concatenate([1.0 + np.arange(8192) / 8192.0, rng.uniform(1.0, 2.0, size=8192),
                        np.ldexp(rng.uniform(1.0, 2.0, size=4096), rng.integers(-1000, 1000, size=4096)),
                        np.nextafter([1.0, 2.0, 4.0], [2.0, 1.0, 3.0])])
    v[::3] *= -1.0
    x, y = torch.from_numpy(v).cuda(), torch.empty(len(v), dtype=torch.float64, device="cuda")
    C.check(C.load().btrt_probe_recip(ctypes.c_void_p(torch.cuda.current_stream().cuda_stream),
                                      ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()), len(v)))
    for a, b in zip(v.tolist(), y.cpu().tolist()):
        assert abs(Fraction(a) * Fraction(b) - 1) <= Fraction(1, 2 ** 52)
