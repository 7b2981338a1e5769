"""Host-side accounting of bench.py (no GPU): the algorithmic bytes per launch follow the union-over-the-
group definition, and the roofline fractions are bytes / time / peak."""
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402
from workloads import WorkloadSpec  # noqa: E402


def _spec():
    return WorkloadSpec(name="acc", config=9, batch=2, n_q_heads=4, n_kv_heads=2, P=3, K_c=5, seq_lens=(100, 40))


def test_union_bytes_count_each_page_and_row_once_per_group():
    spec = _spec()
    sl = np.array([100, 40])                       # 7 and 3 pages
    # routed pages [B, Hq, P]: heads 0,1 form group 0, heads 2,3 group 1
    rp = np.array([[[0, 1, 2], [1, 2, 3], [5, 6, -1], [5, 6, -1]],
                   [[0, 1, -1], [0, 1, -1], [2, -1, -1], [1, 2, -1]]])
    # candidate positions [B, Hq, K_c]
    cp = np.array([[[0, 1, 2, 3, 4], [3, 4, 5, 6, 7], [80, 81, -1, -1, -1], [80, 82, -1, -1, -1]],
                   [[0, 1, 2, 3, 4], [0, 1, 2, 3, 4], [33, -1, -1, -1, -1], [17, 33, -1, -1, -1]]])
    fb = np.array([[0, 1, 0, 0], [0, 0, 0, 0]])
    a = bench.algorithmic_bytes(spec, sl, rp, cp, fb)
    union_pages = 4 + 2 + 2 + 2                     # {0,1,2,3}, {5,6}, {0,1}, {1,2}
    union_rows = 8 + 3 + 5 + 2                      # {0..7}, {80,81,82}, {0..4}, {17,33}
    assert a["sparse_union_pages"] == union_pages and a["sparse_union_rows"] == union_rows
    units = 8
    assert a["sparse_decode"] == union_pages * 16 * 256 + union_rows * 256 + units * (256 + 512)
    # scan: one 256-byte summary row per (page, KV head) + a block-table entry per page + q
    assert a["route_scan"] == (7 + 3) * (2 * 256 + 4) + units * 256
    # a sparse kernel that scans the pages itself: the scan's bytes are its own, q counted once
    b = bench.algorithmic_bytes(spec, sl, rp, cp, fb, scan_inside=True)
    scan = a["route_scan"] - units * 256
    assert "route_scan" not in b and b["sparse_decode"] == a["sparse_decode"] + scan
    assert b["sparse_decode_per_head_model"] == a["sparse_decode_per_head_model"] + scan
    # dense: K and V rows of every (sequence, KV head) with a flagged head
    assert a["dense_fallback"] == 100 * 2 * 256
    # the paper's per-query-head model books every head's pages and rows
    per_head = ((3 * 16 + 5) * 256) * 4 + ((3 * 16 + 5) * 256) * 4 + units * 768
    assert a["sparse_decode_per_head_model"] == per_head


def test_fractions_are_bytes_over_time_over_peak():
    alg = {"route_scan": 10_000_000, "sparse_decode": 5_000_000, "sparse_decode_per_head_model": 20_000_000,
           "dense_fallback": 0}
    pk = {"route_scan": 10.0, "event_pair_overhead": 2.0, "sparse_decode": 5.0, "dense_fallback": 1.0}
    k = bench.kernel_fracs(alg, pk, 12.5, 5000.0)
    assert abs(k["route_scan"]["achieved_GBps"] - 1000.0) < 1e-9 and abs(k["route_scan"]["frac"] - 0.2) < 1e-12
    assert abs(k["sparse_decode"]["frac"] - 0.2) < 1e-12 and abs(k["sparse_decode"]["frac_per_head_model"] - 0.8) < 1e-12
    assert abs(k["step"]["achieved_GBps"] - 15_000_000 / 12.5e-6 / 1e9) < 1e-9
    assert abs(k["sparse_decode"]["frac_of_8TBps"] - 1000.0 / 8000.0) < 1e-12


@pytest.mark.parametrize("head_dim", [64, 128, 256])
def test_step_buffers_and_copied_bytes_follow_the_head_dimension(head_dim):
    from paper_2602_13804_b200 import binding as B
    shape = B.make_shape(3, 8, 2, 5, 20, head_dim=head_dim)
    out, diag, routed, flist, fcount = bench.step_buffers(shape, 7, "cpu")
    assert out.shape == (3, 8, head_dim) and out.element_size() == 4
    assert diag.numel() * diag.element_size() == 24 * B.DIAG_BYTES
    assert routed.shape == (3, 8, 7) and flist.shape == (24,) and fcount.shape == (1,)
    import torch
    q = torch.empty((3, 8, head_dim), dtype=torch.bfloat16)
    assert bench.e2e_bytes(2, q, out, diag) == (2 * 24 * head_dim * 2, 2 * 24 * (head_dim * 4 + 32))


def test_harness_allocates_what_the_step_writes(monkeypatch):
    """The harness of a head-dimension-256 workload, built on the CPU with the library call left out."""
    import torch
    from dataclasses import replace
    from paper_2602_13804_b200 import binding as B
    monkeypatch.setattr(B, "vsa_build_page_summaries", lambda *a, **k: None)
    monkeypatch.setattr(torch.cuda, "mem_get_info", lambda dev=None: (1 << 34, 1 << 34))
    monkeypatch.setattr(torch.cuda, "synchronize", lambda *a: None)
    monkeypatch.setattr(torch.cuda, "Stream", lambda *a, **k: None)

    class Event:
        def __init__(self, **k): pass
        def record(self, *a): pass
        def elapsed_time(self, other): return 0.0
    monkeypatch.setattr(torch.cuda, "Event", Event)
    for d in (64, 128, 256):
        h = bench.Harness(replace(_spec(), head_dim=d, layers=2), torch.device("cpu"))
        assert h.out.numel() == h.units * d and h.summaries[0].shape[-1] == d and h.layers[0].q.shape[-1] == d


def test_the_line_on_stdout_keeps_what_is_asked_for_and_stays_short():
    """A record of the default run, with the longest texts that its fields take, as one line of at most LINE_LIMIT characters."""
    import json
    x = 12345.678901234567
    path = ("route -> sparse with routing certificate -> retries of the refused units with up to 1024 pages -> dense fallback")
    record = {
        "metric": bench.METRIC, "value": x, "unit": bench.UNIT, "n_gpus": 8, "steps": 1000, "warmup": 100, "ms_per_step": x,
        "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "cfg2_b16_t131072_P1024_Kc1024_per_qhead_round_robin", "batch": 64, "n_q_heads": 64, "n_kv_heads": 32,
                   "head_dim": 256, "page_size": 16, "context": 131072, "P": 1024, "K_c": 1024, "epsilon": x, "gap_threshold": x,
                   "layers_per_step": 32, "distinct_layer_caches": 32,
                   "l2": "inputs larger than L2: 32 distinct layer caches, 123456 MB touched per pass over them",
                   "launch": "cuda graph replay of the whole step", "path": path},
        "sustained": {"steps": 1, "note": "n" * 200}, "kernels": {"route_scan": "k" * 1000}, "gpu_launches": 123456,
        "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "power_w_max": x, "reasons": ["sw_power_cap"], "samples": 5},
        "e2e": {"value": x, "unit": bench.UNIT, "ms_per_step": x, "h2d_bytes_per_step": 1 << 30, "d2h_bytes_per_step": 1 << 30,
                "api": "a" * 200},
        "roofline": {"bound": "hbm", "achieved": x, "peak": x, "unit": "GB/s", "frac": x / 1e5, "traffic": x * 1e6,
                     "kernel": "dense_fallback", "us_is": "u" * 400},
        "cpu_baseline": {"value": x, "unit": bench.UNIT, "cores": 128, "kind": "oracle",
                         "sample": "one layer of 32, all 64 sequences, 200 repetitions of one oracle decode step (summaries "
                                   "prebuilt)", "extra_samples": "e" * 300},
        "sweep": {"points": ["s" * 17000]},
    }
    text = bench.short_line(record)
    line = json.loads(text)
    assert len(text) <= bench.LINE_LIMIT and "\n" not in text
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
                "dtype", "data", "gpu_launches"):
        assert line[key] == record[key]
    assert line["e2e"]["value"] == x and line["clocks"]["reasons"] == ["sw_power_cap"] and line["cpu_baseline"]["cores"] == 128
    assert line["config"]["l2"] == record["config"]["l2"] and line["roofline"]["frac"] == record["roofline"]["frac"]
    assert bench.short_line({**record, "e2e": None, "cpu_baseline": None})       # variants without an end-to-end form
