"""FP64 lattices at the ends of the integer collision's range (csrc/btrt_fx.cuh),
against the FP64 oracle: fields whose nodes pull nine (nineteen) equal populations at
the top of a binade, the largest sums a node can form."""
import numpy as np
import pytest

import oracle
import workloads as w
from conftest import cpu_threads
from oracle import d3q19 as o3

pytestmark = pytest.mark.gpu

TOL64 = 1e-11


def _rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def _check2(p, steps):
    from paper_1902_09813_gb300 import Lattice
    lat = Lattice.from_problem(p, compute="f64").init(p.phi0(), t0=p.t0)
    ref = oracle.OracleLattice(p, nthreads=cpu_threads()).init()
    for n in steps:
        lat.step(n)
        ref.step(n)
    phi = ref.phi()
    ref.step(1)
    assert _rel(lat.phi_host(), phi) <= TOL64
    assert _rel(lat.read_f(), ref.fpost) <= TOL64
    assert lat.check() == 0


def _check3(p, steps):
    from paper_1902_09813_gb300 import Lattice3
    lat = Lattice3.from_problem(p, compute="f64").init(p.phi0()).step(steps)
    ref = o3.OracleLattice3(p, nthreads=cpu_threads()).init()
    ref.step(steps)
    phi = ref.phi()
    ref.step(1)
    assert _rel(lat.phi_host(), phi) <= TOL64
    assert _rel(lat.read_f(), ref.fpost) <= TOL64
    assert lat.check() == 0


COEFFS = {"linear": dict(), "general": dict(b2=1e-3, c3=1e-3, a2=0.1), "reaction": dict()}


def _with(p, kind, k0):
    p = p.replace(u=(0.0,) * len(p.u), k0=k0, k2_mode="const", k2=k0, **COEFFS[kind])
    if kind == "reaction":
        p.source.kind, p.source.const, p.source.exp = "reaction", 0.01, 2.0
    return p


@pytest.mark.parametrize("steps", [(1,), (3,)], ids=["one", "three"])
@pytest.mark.parametrize("kind", COEFFS)
@pytest.mark.parametrize("k0", [1.6, 1.9, 1.99])
def test_equal_populations(kind, k0, steps):
    p = w.random_state_problem(34, 32, seed=2, nonlinear=False, source="none")
    x, y = np.arange(34)[None, :] % 2, np.arange(32)[:, None] % 2
    a = (1.0 / k0 - 0.5) / 3.0                       # K1 = k0 I
    p = _with(p.replace(A0=(a, 0.0, a), phi0_array=4.49 / 128 * 4.0 ** (x + y)), kind, k0)
    _check2(p, steps)


@pytest.mark.parametrize("kind", COEFFS)
@pytest.mark.parametrize("k0", [1.6, 1.9, 1.99])
def test_equal_populations_d3q19(kind, k0):
    p = w.random_state_problem3(12, 10, 8, seed=2, nonlinear=False, source="none")
    n = (np.arange(12)[None, None, :] % 2) + (np.arange(10)[None, :, None] % 2) + (np.arange(8)[:, None, None] % 2)
    a = (1.0 / k0 - 0.5) / 3.0
    field = 3 * 1.99 / 64 * np.array([1.0, 6.0, 12.0, 12.0])[n]
    p = _with(p.replace(A0=(a, 0.0, 0.0, a, 0.0, a), phi0_fn=lambda X, Y, Z: field), kind, k0)
    _check3(p, 2)


@pytest.mark.parametrize("u", [(0.45, 0.52), (-0.55, 0.3), (0.7, -0.95)], ids=str)
@pytest.mark.parametrize("k0", [1.0, 1.2])
@pytest.mark.parametrize("size", [(41, 33), (37, 29)], ids=["many-steps", "plain"])
def test_fast_flow(u, k0, size):
    """Per-node coefficients with half a cell and more per step."""
    p = w.random_state_problem(*size, seed=4, bc=(0, 0, 1, 1), nonlinear=True, source="trig").replace(u=u, k0=k0)
    _check2(p, (5,))


@pytest.mark.parametrize("nonlinear", [False, True])
@pytest.mark.parametrize("dim", [2, 3])
def test_tiny_values(dim, nonlinear):
    """A field around 1e-300, with zeros: the relative accuracy of ordinary values."""
    n, draw = ((48, 37), w.random_state_problem) if dim == 2 else ((12, 11, 9), w.random_state_problem3)
    p = draw(*n, seed=6, nonlinear=nonlinear, source="none")
    field = 1e-300 * p.phi0()
    field[..., :5] = 0.0
    if dim == 2:
        from paper_1902_09813_gb300 import Lattice as L
        ref = oracle.OracleLattice(p.replace(phi0_array=field), nthreads=cpu_threads()).init()
    else:
        from paper_1902_09813_gb300 import Lattice3 as L
        ref = o3.OracleLattice3(p.replace(phi0_fn=lambda X, Y, Z: field), nthreads=cpu_threads()).init()
    lat = L.from_problem(p, compute="f64").init(field).step(3)
    ref.step(3)
    assert lat.check() == 0
    assert _rel(lat.phi_host() * 2.0 ** 990, ref.phi() * 2.0 ** 990) <= TOL64
    ref.step(1)
    assert _rel(lat.read_f() * 2.0 ** 990, ref.fpost * 2.0 ** 990) <= TOL64
