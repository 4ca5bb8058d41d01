"""D3Q19 with 16-bit storage: large constant-coefficient lattices take two nodes per
thread, small ones a node per thread, with the same arithmetic.  A z-periodic problem
repeated along z crosses the size where the form changes and must repeat bit for
bit."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("shift", ["local", "ref"])
@pytest.mark.parametrize("nx,ny,bc", [(52, 26, (0, 0, 0, 0, 0, 0)), (51, 26, (0, 0, 1, 1, 0, 0)), (65, 21, (1, 1, 0, 0, 0, 0)),
                                      (66, 21, (1, 1, 1, 1, 0, 0)), (130, 12, (0, 0, 0, 0, 0, 0))],
                         ids=["even", "odd-ywalls", "odd-xwalls", "even-walls", "wide"])
@pytest.mark.parametrize("source", ["none", "const"])
@pytest.mark.parametrize("k0", [1.0, 1.1])
def test_repeated_along_z(storage, shift, nx, ny, bc, source, k0):
    from paper_1902_09813_gb300 import Lattice3
    nz = 80
    p = w.random_state_problem3(nx, ny, nz, seed=9, bc=bc, nonlinear=False, source=source).replace(k0=k0)
    assert nx * ny * nz < 1 << 17 <= 2 * nx * ny * nz
    phi0 = p.phi0()
    a = Lattice3.from_problem(p, compute="f32", storage=storage, shift=shift).init(phi0).step(7)
    b = Lattice3.from_problem(p.replace(nz=2 * nz), compute="f32", storage=storage, shift=shift)
    b.init(np.concatenate([phi0, phi0])).step(7)
    assert a.check() == 0 and b.check() == 0
    pa, pb = a.phi_host(), b.phi_host()
    assert np.array_equal(pb[:nz], pa) and np.array_equal(pb[nz:], pa)
    fa, fb = a.read_f(), b.read_f()
    assert np.array_equal(fb[:, :nz], fa) and np.array_equal(fb[:, nz:], fa)
