"""The step whose sparse pass scans the pages itself (small batches of short contexts), beside its limits: tables whose tiles
just fill a block's share and one page more (with and without blocks that only help with the scan), every group size, ragged
lengths down to one page, and entries of the table that name no page.  Compared with the oracle and with the separate calls."""
import numpy as np
import pytest

from gpu_runner import compare, run_gpu
from test_gpu_fp8 import compare as _compare, run_fp8
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu


def _workload(batch, hq, hkv, pages, d=128, page=16, P=12, K_c=60):
    lens = (page * pages - 3,) + tuple(1 + (page * pages * i) // (batch + 1) for i in range(1, batch))
    return make_workload(WorkloadSpec(name="scan", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, P=P, K_c=K_c,
                                      seq_lens=lens, needles=2, needle_positions="uniform", page_size=page), seed=8800 + pages + hq)


@pytest.mark.parametrize("batch,hq,hkv,pages,d,page", [
    (1, 32, 8, 256, 128, 16),    # four blocks to a cluster, or eight
    (1, 32, 8, 257, 128, 16),
    (1, 32, 8, 512, 128, 16),
    (1, 32, 8, 513, 128, 32),    # scanned ahead
    (4, 32, 8, 256, 128, 16),    # 128 units
    (5, 32, 8, 17, 128, 16),     # 160: scanned ahead
    (2, 64, 8, 1024, 128, 16),   # eight heads, more rounds than one; 128 units: scanned ahead
    (1, 64, 8, 1024, 128, 16),
    (1, 64, 8, 1025, 128, 16),
    (3, 16, 1, 300, 128, 16),    # sixteen heads: two clusters to a KV head
    (2, 32, 1, 31, 64, 32),
    (2, 8, 8, 256, 128, 16),     # one head: clusters of one block and of helpers
    (2, 8, 8, 2048, 128, 16),
    (3, 6, 3, 1023, 128, 16),
    (1, 32, 8, 512, 64, 16),
    (1, 32, 8, 1025, 64, 16),
    (1, 32, 8, 128, 256, 16),
    (2, 8, 2, 257, 256, 32),
    (7, 4, 2, 1, 128, 16),       # one page
])
def test_scan_in_the_sparse_pass(batch, hq, hkv, pages, d, page):
    w = _workload(batch, hq, hkv, pages, d, page)
    compare(w, run_gpu(w), dense_sample=2)
    g = run_gpu(w, gap_threshold=float("inf"))      # every unit with a rejected token falls back
    compare(w, g, gap_threshold=float("inf"), dense_sample=2)


def test_fp8():
    _compare(*run_fp8(_workload(2, 8, 2, 300)))


def test_bad_pages_and_lengths():
    w = _workload(3, 8, 2, 100).to("cuda:0")
    ref = run_gpu(w)
    w.block_table[0, 5] = w.k_cache.shape[0] + 7
    w.block_table[0, 99] = -1
    w.seq_lens[1] = 0
    got = run_gpu(w, summaries=ref.summaries)
    assert np.array_equal(got.step_routed, got.routed_pages) and np.array_equal(got.step_out, got.out)
    for name in got.step_diag:
        assert np.array_equal(got.step_diag[name], got.diag[name], equal_nan=True), name
    assert np.array_equal(got.step_out[2], ref.step_out[2])
    assert (got.step_diag["status"].reshape(3, 8)[1] != 0).all() and not got.step_diag["status"].reshape(3, 8)[0].any()
