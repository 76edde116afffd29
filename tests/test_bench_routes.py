"""bench.py's kernel report on made-up counters: a solve whose inner solves run in one launch is reported as that
one kernel with its own traffic and no fraction of the HBM peak, and the multilevel bytes follow the
deflation rank at which the post-smoothing leaves the gather."""
import math

import bench


def _stats(**kw):
    st = {"inner_phase1_timed": 1000, "inner_phase1_csum": 4000, "inner_phase1_ms": 6.0, "inner_rows_ms": 1.5,
          "inner_phase2_ms": 2.5, "n_long_rows": 0, "sell_entries": 40320, "precond": 0, "ml_coarse_n": 300,
          "ml_coarse_nnz": 2000}
    st.update(kw)
    return st


def _route(ctas=0, staged=0):
    return {"one_launch_ctas": ctas, "staged": staged, "renumbered": 0}


def test_one_launch_solve_is_one_kernel():
    n = 10000
    out, dom, _ = bench.kernel_rooflines(_stats(), n, 39600, 4, "grid100x100", "f32", [_route(16)] * 5)
    assert dom == "one_launch" and list(out) == ["one_launch"]
    e = out[dom]
    assert "k_minres_cluster" in e["kernel"] and "k_phase1" not in e["kernel"]
    assert e["frac"] is None and e["peak"] is None and e["bound"] == "latency"
    assert math.isclose(e["avg_us"], 10.0) and math.isclose(e["total_ms"], 10.0)
    assert e["bytes_per_launch"] == 8 * 40320 + 16 * 313 + 4 * n + 2 * 4 * 4 * n
    staged, _, _ = bench.kernel_rooflines(_stats(), n, 39600, 4, "x", "f32", [_route(16, 1)] * 5)
    assert staged["one_launch"]["bytes_per_launch"] == 4 * 40320 + 16 * 313 + 17 * 4 * n + 2 * 4 * 4 * n


def test_ranks_that_leave_the_one_launch_solve_are_named():
    out, _, _ = bench.kernel_rooflines(_stats(), 10000, 39600, 8, "x", "f64", [_route(16)] * 3 + [_route()] * 2)
    assert "ranks 3, 4 take" in out["one_launch"]["kernel"]


def test_launches_per_iteration_keep_three_kernels():
    out, _, _ = bench.kernel_rooflines(_stats(), 10000, 39600, 4, "x", "f32", [_route()] * 5)
    assert list(out) == ["gather", "rows", "phase2"] and out["gather"]["bound"] == "hbm"


def test_multilevel_bytes_follow_the_rank():
    n, Z, w = 100000, 400000, 4
    st = _stats(precond=1)
    few, _, _ = bench.kernel_rooflines(st, n, Z, w, "x", "f32", [_route()] * 9)
    many, _, _ = bench.kernel_rooflines(st, n, Z, w, "x", "f32", [_route()] * 18)
    ns = (n + 31) // 32
    fused = bench.kernel_bytes("phase2_ml_s", n, Z, 4.0, w, 0, ns, (300, 2000))
    assert few["phase2"]["bytes_per_launch"] == fused
    assert math.isclose(many["phase2"]["bytes_per_launch"], fused + 3 * w * n / 2)
