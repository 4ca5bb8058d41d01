"""Many steps per launch (the default of small lattices) against one step per launch:
the same arithmetic in the same order, so the fields and populations are equal bit
for bit -- over stored forms, boundaries, sources, tile remainders and step counts
that end within a round or go over one launch."""
import numpy as np
import pytest

import workloads as w

pytestmark = pytest.mark.gpu

FORMS = [("f64", "f64", "ref"), ("df64", "df64", "ref"), ("f32", "f32", "ref"), ("f32", "f32", "local"),
         ("f32", "f16", "local"), ("f32", "f16", "ref"), ("f32", "bf16", "local"), ("f32", "f16", "local_sr"),
         ("f32", "bf16", "local_sr"), ("f32", "f32", "local_dw"), ("f32", "bf16", "local_dw_sr"),
         ("f32", "bf16", "moment_sr"), ("f32", "f16", "moment_sr")]


def _pair(p, form, steps):
    from paper_1902_09813_gb300 import Lattice
    out = []
    for variant in ("auto", "plain"):
        lat = Lattice.from_problem(p, compute=form[0], storage=form[1], shift=form[2])
        lat.set_sweep_variant(variant)
        lat.init(p.phi0(), t0=p.t0)
        for n in steps:
            lat.step(n)
        assert lat.check() == 0 and lat.time()[0] == sum(steps)
        out.append((lat.phi_host(), lat.read_f()))
    return out


def _same(p, form, steps):
    (phi_a, f_a), (phi_b, f_b) = _pair(p, form, steps)
    assert np.array_equal(phi_a, phi_b)
    assert np.array_equal(f_a, f_b)


@pytest.mark.parametrize("form", FORMS, ids=lambda f: "-".join(f))
@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 1, 1, 1), (1, 1, 0, 0), (0, 0, 1, 1)], ids=str)
@pytest.mark.parametrize("nonlinear", [False, True])
def test_equal_to_one_step_per_launch(form, bc, nonlinear):
    p = w.random_state_problem(61, 43, seed=3, bc=bc, nonlinear=nonlinear, source="trig")
    _same(p, form, (11,))


@pytest.mark.parametrize("form", FORMS[:1] + FORMS[2:3] + FORMS[4:5], ids=lambda f: "-".join(f))
@pytest.mark.parametrize("size", [(32, 32), (33, 40), (48, 49), (96, 32), (130, 65), (256, 255)], ids=str)
def test_tile_remainders(form, size):
    p = w.random_state_problem(*size, seed=5, bc=(0, 0, 1, 1), nonlinear=False, source="const")
    _same(p, form, (9, 2, 4, 5))


@pytest.mark.parametrize("form", FORMS[:3] + FORMS[4:5], ids=lambda f: "-".join(f))
@pytest.mark.parametrize("steps", [(2,), (3,), (1, 4, 1), (7, 8), (257,), (258, 255)], ids=str)
def test_step_counts(form, steps):
    p = w.random_state_problem(40, 36, seed=6, bc=(1, 1, 0, 0), nonlinear=False, source="trig")
    _same(p, form, steps)


@pytest.mark.parametrize("form", FORMS[:1] + FORMS[2:3] + FORMS[4:5], ids=lambda f: "-".join(f))
def test_reaction_source_fields_and_wall_arrays(form):
    p = w.burgers_fisher(n=48)
    walls = p.wall_arrays_at(0.0)
    _same(p.replace(wall_fn=None, wall_arrays=walls), form, (13,))
    _same(w.variable_tensor(n=50), form, (13,))
    _same(w.linear_cde(n=44, walls=True), form, (13,))


def test_residual_and_non_finite_flag():
    from paper_1902_09813_gb300 import Lattice
    from paper_1902_09813_gb300 import _capi as C
    p = w.steady_diffusion(n=40)
    a, b = (Lattice.from_problem(p, compute="f64").init(p.phi0()) for _ in range(2))
    b.set_sweep_variant("plain")
    assert a.step_residual(22) == b.step_residual(22)
    phi0 = p.phi0()
    phi0[7, 9] = np.nan
    a.init(phi0).step(6)
    with pytest.raises(C.BtrtError):
        a.check()


@pytest.mark.parametrize("size", [(49, 33), (50, 41), (32, 400), (700, 33), (97, 57)], ids=str)
@pytest.mark.parametrize("form", FORMS[:1] + FORMS[2:3] + FORMS[-1:], ids=lambda f: "-".join(f))
def test_narrow_last_tiles(size, form):
    """Last tiles of one to a few nodes: a region then reaches over them into the next
    tile, on periodic axes round the lattice."""
    p = w.random_state_problem(*size, seed=8, nonlinear=False, source="none")
    _same(p, form, (41,))


@pytest.mark.parametrize("size", [(723, 725), (513, 512), (130, 4001)], ids=str)
def test_largest_double_word_phi(size):
    p = w.random_state_problem(*size, seed=9, bc=(1, 1, 0, 0), nonlinear=False, source="trig")
    _same(p, ("f32", "f32", "local_dw"), (9,))
