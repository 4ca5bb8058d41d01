"""Many steps per launch: a refused cooperative launch, and a grid barrier that gives up."""
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

import workloads as w
from conftest import ROOT

pytestmark = pytest.mark.gpu

# cudaLaunchCooperativeKernel that answers cudaErrorCooperativeLaunchTooLarge and launches nothing
FAKE = r"""
#include <stdio.h>
int cudaLaunchCooperativeKernel(const void *f, ...) {
    (void)f;
    fprintf(stderr, "refused\n");
    return 720;
}
"""
RUN = r"""
import sys
sys.path[:0] = [%r, %r]
import numpy as np
import workloads as w
from paper_1902_09813_gb300 import Lattice
for form in (("f64", "f64", "ref"), ("df64", "df64", "ref"), ("f32", "f32", "ref"), ("f32", "f16", "local"),
             ("f32", "bf16", "moment_sr")):
    p = w.random_state_problem(61, 43, seed=3, bc=(0, 0, 1, 1), nonlinear=True, source="trig")
    out = []
    for variant in ("auto", "plain"):
        lat = Lattice.from_problem(p, compute=form[0], storage=form[1], shift=form[2])
        lat.set_sweep_variant(variant)
        lat.init(p.phi0(), t0=p.t0).step(11).step(2)
        assert lat.check() == 0 and lat.time()[0] == 13
        out.append((lat.phi_host(), lat.read_f()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
print("equal")
"""


def test_refused_cooperative_launch(tmp_path):
    """A context with fewer SMs than the device (an MPS share, a green context) refuses the launch:
    the lattice then advances in the other forms, bitwise the same."""
    cc = shutil.which("gcc")
    if cc is None:
        pytest.skip("no gcc")
    (tmp_path / "fake.c").write_text(FAKE)
    so = tmp_path / "fake.so"
    subprocess.run([cc, "-shared", "-fPIC", str(tmp_path / "fake.c"), "-o", str(so)], check=True)
    r = subprocess.run([sys.executable, "-c", RUN % (ROOT, os.path.join(ROOT, "tests"))], capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=str(so)), timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    assert "equal" in r.stdout and r.stderr.count("refused") >= 5


@pytest.mark.parametrize("form", [("f64", "f64", "ref"), ("f32", "f32", "ref"), ("f32", "f16", "local")], ids="-".join)
def test_barrier_that_gives_up(form):
    """Blocks that find the others not yet there and may not wait: the launch ends, the check
    says so, and a new initial field makes the lattice usable again."""
    from paper_1902_09813_gb300 import Lattice
    from paper_1902_09813_gb300 import _capi as C
    p = w.random_state_problem(120, 90, seed=7, nonlinear=False, source="trig")
    lat, ref = (Lattice.from_problem(p, compute=form[0], storage=form[1], shift=form[2]) for _ in range(2))
    lat.set_wait_limit(0)
    lat.init(p.phi0(), t0=p.t0).step(64)
    with pytest.raises(C.BtrtError) as err:
        lat.check()
    assert err.value.code == C.ETIMEOUT and lat.flags() & 4
    lat.set_wait_limit(1 << 22)
    lat.init(p.phi0(), t0=p.t0).step(64)
    ref.set_sweep_variant("plain")
    ref.init(p.phi0(), t0=p.t0).step(64)
    assert lat.check() == 0
    assert np.array_equal(lat.phi_host(), ref.phi_host()) and np.array_equal(lat.read_f(), ref.read_f())


@pytest.mark.parametrize("size,form,nonlinear", [
    ((181, 181), ("f64", "f64", "ref"), False), ((131, 187), ("f64", "f64", "ref"), True),
    ((255, 257), ("df64", "df64", "ref"), False), ((181, 181), ("df64", "df64", "ref"), True),
    ((363, 361), ("f32", "f32", "ref"), True), ((33, 3971), ("f32", "f32", "local"), False),
    ((511, 513), ("f32", "f16", "local"), True), ((8191, 32), ("f32", "bf16", "ref"), False),
    ((511, 513), ("f32", "bf16", "moment_sr"), False), ((509, 515), ("f32", "f16", "local_sr"), True),
    ((100, 2621), ("f32", "f16", "moment_sr"), True), ((511, 513), ("f32", "bf16", "local_dw_sr"), True),
    ((49, 33), ("df64", "df64", "ref"), False), ((32, 49), ("df64", "df64", "ref"), True)],
    ids=lambda v: "-".join(map(str, v)) if isinstance(v, tuple) else ("nonlinear" if v else "linear"))
def test_largest_sizes(size, form, nonlinear):
    """The largest lattices of the rule, with ragged tiles and more tiles than are resident: equal to
    one step per launch bit for bit, and the many-steps form is the one that runs."""
    from paper_1902_09813_gb300 import Lattice
    from paper_1902_09813_gb300.lattice import auto_form
    p = w.random_state_problem(*size, seed=12, bc=(0, 0, 1, 1), nonlinear=nonlinear, source="trig")
    out = []
    for variant in ("auto", "plain"):
        lat = Lattice.from_problem(p, compute=form[0], storage=form[1], shift=form[2])
        assert auto_form(lat.desc, nonlinear) == "many"
        lat.set_sweep_variant(variant)
        lat.init(p.phi0(), t0=p.t0).step(11)
        assert lat.check() == 0
        out.append((lat.phi_host(), lat.read_f()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
