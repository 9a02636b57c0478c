"""Which kernels the benchmark names for a workload's query, and that it derives requests per second from
the markers only where they count reads (not along a walk, whose cells serve many coordinates)."""

import bench


def test_names_and_counts():
    big = 1 << 25
    assert bench.query_kernels(5, 1 << 18, big) == ("k_qsample + k_pbits + k_query_bits<5> + k_repair", True)
    assert bench.query_kernels(7, 1 << 20, big) == ("k_qsample + k_query_walk<7> (or k_query<7>) + k_repair", False)
    assert bench.query_kernels(10, 1 << 20, big) == ("k_qsample + k_query<10> + k_repair", True)
    assert bench.query_kernels(5, 1 << 20, 1 << 20) == ("k_query<5>", True)
    assert bench.query_kernels(5, 30_011, big) == ("k_query_mod<5>", True)


def test_walk_reports_no_request_rate():
    class Workload:
        P, d, r, c, k, name = 8, 1 << 25, 7, 1 << 20, 1 << 15, "x"

    class Run:
        w, main_rows, groups, insert_launches, staged, W, use_plan = Workload, 1, 1, 2, False, 8, True

    ph = {"insert": 1.0, "query": 0.5, "select": 0.1, "query_select": None, "n": 1}
    _, q = bench.rooflines(Run, "error_feedback", ph, {"hbm_gbs": 6780.0}, "measured", {"query_ms": 0.6}, 0.9, 4.5, 4.5)
    for key in ("requests_per_step", "achieved_G_requests_per_s", "requests_frac_of_ceiling", "cells_read_per_coord"):
        assert q[key] is None, key
    assert q["time_vs_full_read_ceiling"] == 1.2
    Workload.r, Workload.c = 5, 1 << 18
    _, q = bench.rooflines(Run, "error_feedback", ph, {"hbm_gbs": 6780.0}, "measured", {"query_ms": 0.6}, 0.9, 3.2, 0.4)
    assert q["requests_frac_of_ceiling"] > 0 and "k_query_bits<5>" in q["kernel"]
