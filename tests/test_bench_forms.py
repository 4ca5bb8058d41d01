"""bench.py's kernel forms follow the library's choice, and its JSON line reports the
roofline that binds."""
import argparse
import json

import bench
import pytest


def _args(**kw):
    a = dict(compute="f64", storage="f64", workload="mms", shift="auto", sweep="auto", steps=1000, n=8192)
    a.update(kw)
    return argparse.Namespace(**a)


@pytest.mark.parametrize("kw,form,launches", [
    (dict(n=64), "many", 4), (dict(n=64, steps=257), "many", 2), (dict(n=182), "plain", 1000),
    (dict(n=157, workload="nonlinear"), "plain", 1000), (dict(n=156, workload="nonlinear"), "many", 4),
    (dict(compute="f32", storage="f32", shift="local_dw", n=513), "many", 4),
    (dict(compute="f32", storage="f32", shift="local_dw", n=724), "many", 4),
    (dict(compute="f32", storage="f32", shift="local_dw", n=725), "plain", 1000),
    (dict(compute="f32", storage="f32", shift="local_dw", n=513, workload="nonlinear"), "plain", 1000),
    (dict(compute="f32", storage="f16", n=512), "many", 4), (dict(compute="f32", storage="f16", n=513), "tb2", 500),
    (dict(compute="f32", storage="bf16", shift="moment_sr", n=1024), "vec", 1000),
    (dict(compute="f32", storage="f32", sweep="tb2", steps=7), "tb2", 4)])
def test_form_and_launches(kw, form, launches):
    a = _args(**kw)
    assert bench.kernel_form(a) == form and bench.launches(a) == launches


@pytest.mark.parametrize("compute,storage", [("f64", "f64"), ("f32", "f16")])
def test_many_steps_have_no_traffic_of_the_one_step_kernel(compute, storage):
    r = bench.binding_roofline(bench.roofline(_args(n=128, compute=compute, storage=storage), 128 * 128, 4e-3, 900.0, 6800.0,
                                              "measured"))
    assert r["kernel"].startswith("sweep_tbn_kernel") and r["traffic"] is None and r["bound"] == "hbm"


def test_fp64_line_reports_hbm():
    nodes, t = 8192 * 8192, 1.75e-3
    r = bench.binding_roofline(bench.roofline(_args(), nodes, t, 160 * nodes / t / 1e9, 6800.0, "measured"))
    assert r["bound"] == "hbm" and r["unit"] == "GB/s" and r["frac"] < 1.0
    assert r["traffic"] == round(bench.FP64_TRAFFIC_PER_NODE * nodes) and r["kernel"].startswith("sweep_kernel")
    assert r["fp64_scheme_view"]["ops_per_update"] == bench.FP64_OPS_PER_UPDATE_LINEAR


def test_line_stays_short():
    """The tables of a full run go beside the line, which keeps every contract key."""
    contract = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline", "batched")
    line = {k: {"filler": "x" * 120} for k in contract}
    line["variants"] = {f"variant_{k}": {"mlups": 1e5, "ms_per_step": 0.5, "algorithmic_gbs": 6e3, "hbm_frac": 0.9}
                        for k in range(70)}
    line["variants"].update({k: {"mlups": 123456.7} for k in bench.LINE_VARIANTS})
    line["accuracy"] = {t: {f"form_{k}": 1e-5 for k in range(16)} for t in
                        ("nonlinear_2048_1000_rel_l2", "nonlinear_8192_1000_rel_l2", "hill_64_gre", "mms_128_gre")}
    rate = {"solves_per_s": 29.2, "p50_s": 2.4, "p99_s": 2.6, "gpu_idle_fraction": 0.03,
            "depth_t_active_waiting": [[0.1 * k, k, 96 - k] for k in range(40)]}
    line["serving"] = {"requests_per_rate": 96, "rates": {r: rate for r in ("100", "500", "2000")},
                       "sequential_plain": dict(rate), "served_vs_sequential": {"bitwise_equal": 96}}
    short, details = bench.split_line(line)
    assert len(json.dumps(line)) > 12000 and len(json.dumps(short)) < 6000
    assert all(short[k] == line[k] for k in contract)
    assert details == {k: line[k] for k in ("variants", "accuracy", "serving")}
    assert short["variants_mlups"]["mms_df64"] == 123457 and short["serving"]["rates"]["500"]["p99_s"] == 2.6
    plain, nothing = bench.split_line({k: line[k] for k in contract})
    assert not nothing and plain == {k: line[k] for k in contract}
