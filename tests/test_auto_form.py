"""Which kernel form AUTO takes (btrt_auto_form): many steps per launch on small lattices,
by nodes and, for 16-bit storage, by the waves of tiles that a narrow lattice makes."""
import pytest


@pytest.fixture(scope="module")
def form():
    import paper_1902_09813_gb300 as pkg
    pkg.build()
    from paper_1902_09813_gb300.lattice import auto_form, grid_desc

    def of(nx, ny, compute, storage, shift="ref", per_node=False):
        return auto_form(grid_desc(nx, ny, 1.0, 1.0, compute=compute, storage=storage, shift=shift), per_node)
    return of


@pytest.mark.parametrize("compute,storage,shift,most,most_per_node", [
    ("f64", "f64", "ref", 181, 156), ("df64", "df64", "ref", 256, 181), ("f32", "f32", "ref", 362, 362),
    ("f32", "f16", "local", 512, 512), ("f32", "bf16", "local", 512, 512), ("f32", "f16", "local_sr", 512, 512),
    ("f32", "bf16", "moment_sr", 512, 512), ("f32", "f32", "local_dw", 724, 512)])
def test_squares(form, compute, storage, shift, most, most_per_node):
    for per_node, n in ((False, most), (True, most_per_node)):
        for k in (32, 33, 64, 100, n):
            assert form(k, k, compute, storage, shift, per_node) == "many"
        assert form(n + 1, n + 1, compute, storage, shift, per_node) != "many"
        assert form(31, 40, compute, storage, shift, per_node) != "many"
        assert form(40, 31, compute, storage, shift, per_node) != "many"


@pytest.mark.parametrize("storage", ["f16", "bf16"])
def test_narrow_lattices(form, storage):
    """Measured against the other form: slower where many steps are not taken."""
    for per_node in (False, True):
        for nx, ny in ((32, 8192), (32, 7776), (32, 6808), (32, 5104), (57, 3400), (64, 3400)):
            assert form(nx, ny, "f32", storage, "local", per_node) == "tb2"
        for nx, ny in ((32, 4096), (8192, 32), (57, 4536), (64, 4096), (100, 2552), (200, 1272)):
            assert form(nx, ny, "f32", storage, "local", per_node) == "many"
    for shift in ("local_sr", "moment_sr"):
        for nx, ny in ((32, 4096), (64, 3400), (57, 4536), (128, 2040)):
            assert form(nx, ny, "f32", storage, shift) == "many"
        for nx, ny in ((32, 8192), (32, 5104)):
            assert form(nx, ny, "f32", storage, shift) == "plain"
        for nx, ny in ((128, 1064), (57, 2432), (57, 4536), (100, 2552)):
            assert form(nx, ny, "f32", storage, shift, True) == "many"
        for nx, ny in ((32, 8192), (32, 2672), (57, 1776), (64, 3400), (128, 2040)):
            assert form(nx, ny, "f32", storage, shift, True) == "plain"


def test_large_lattices(form):
    assert form(8192, 8192, "f64", "f64") == "plain"
    assert form(8192, 8192, "f32", "f32") == "tb2"
    assert form(8192, 8192, "f32", "f16", "local") == "vec"
    assert form(1024, 1024, "f32", "f16", "local") == "tb2"
    assert form(1024, 1024, "f32", "bf16", "moment_sr") == "vec"
    assert form(1024, 1024, "f32", "bf16", "moment_sr", True) == "plain"
