"""D3Q19 with 16-bit storage, two nodes per thread: walls on z and the sources that
test_gpu_d3q19_pairs.py leaves out.  A y-periodic problem repeated along y crosses the
size where the form changes and must repeat bit for bit."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("shift", ["local", "ref"])
@pytest.mark.parametrize("source", ["field", "reaction", "none"])
@pytest.mark.parametrize("nx,nz,bc", [(52, 26, (0, 0, 0, 0, 1, 1)), (51, 26, (1, 1, 0, 0, 1, 1)), (65, 21, (0, 0, 0, 0, 0, 0))],
                         ids=["even-zwalls", "odd-xzwalls", "odd-periodic"])
def test_repeated_along_y(storage, shift, source, nx, nz, bc):
    from paper_1902_09813_gb300 import Lattice3
    ny = 80
    p = w.random_state_problem3(nx, ny, nz, seed=9, bc=bc, nonlinear=False, source=source)
    assert nx * ny * nz < 1 << 17 <= 2 * nx * ny * nz
    phi0 = p.phi0()
    q = p.replace(ny=2 * ny)
    if p.src_field is not None:
        q = q.replace(src_field=np.concatenate([p.src_field, p.src_field], axis=1))
    a = Lattice3.from_problem(p, compute="f32", storage=storage, shift=shift).init(phi0).step(7)
    b = Lattice3.from_problem(q, compute="f32", storage=storage, shift=shift)
    b.init(np.concatenate([phi0, phi0], axis=1)).step(7)
    assert a.check() == 0 and b.check() == 0
    pa, pb = a.phi_host(), b.phi_host()
    assert np.array_equal(pb[:, :ny], pa) and np.array_equal(pb[:, ny:], pa)
    fa, fb = a.read_f(), b.read_f()
    assert np.array_equal(fb[:, :, :ny], fa) and np.array_equal(fb[:, :, ny:], fa)
