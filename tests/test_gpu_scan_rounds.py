"""Scans of the pages in clusters of the sparse pass with several tiles of pages to a warp (the copies ahead reuse their stages), for scores
in shared memory and in registers, and under the solves with one block to an SM.  Every shape is checked to take the scan that
it stands for; results as from the separate calls, bit for bit."""
import numpy as np
import pytest
import torch

from gpu_runner import run_gpu
from paper_2602_13804_b200 import binding as B
from test_gpu_page_mma import _keys
from test_gpu_solver import run_entropic, run_fw
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu


def _workload(batch, hq, hkv, table, lens, d=128, page=16, P=24, K_c=100):
    w = make_workload(WorkloadSpec(name="rounds", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, P=P, K_c=K_c,
                                   seq_lens=tuple(lens), needles=2, needle_positions="uniform", page_size=page), seed=9300 + batch + hq)
    w.block_table = torch.nn.functional.pad(w.block_table, (0, table - w.block_table.shape[1]), value=-1)
    return w


def _check(w, scan):
    shape = B.shape_of(w.q, w.k_cache, w.block_table)
    assert B.vsa_step_scan(shape, w.spec.P, w.spec.K_c) == getattr(B, "VSA_STEP_SCAN_" + scan)
    g = run_gpu(w)
    assert np.array_equal(g.step_routed, g.routed_pages)
    for name in g.step_diag:
        if name != "lse":                       # (rewritten by the dense pass where a unit falls back)
            assert np.array_equal(g.step_diag[name], g.diag[name], equal_nan=True), name
    assert np.array_equal(g.step_fallback_units, g.fallback_units)
    units = w.q.shape[0] * w.q.shape[1]
    sparse = np.setdiff1d(np.arange(units), g.fallback_units)
    assert np.array_equal(g.step_out.reshape(units, -1)[sparse], g.out.reshape(units, -1)[sparse])


@pytest.mark.parametrize("kind", ["generated", "equal", "near"])
@pytest.mark.parametrize("batch,hq,hkv,table,longest,d,scan", [
    (4, 32, 8, 4096, 40009, 128, "INSIDE_MMA"),     # 512 threads
    (8, 32, 8, 2100, 33333, 128, "INSIDE_MMA"),     # 256 threads, a block to an SM and a half
    (38, 4, 1, 2100, 33333, 128, "INSIDE_MMA"),     # scores in shared memory
    (38, 4, 1, 4100, 65001, 64, "INSIDE_MMA"),      # eight tiles to a warp, four stages
    (38, 4, 1, 2100, 33333, 256, "INSIDE_MMA"),     # one stage
    (1, 64, 8, 1024, 16001, 128, "INSIDE"),
])
def test_many_pages(batch, hq, hkv, table, longest, d, scan, kind):
    lens = (longest,) + tuple((1, 700, 16 * 33, 4097)[i % 4] for i in range(batch - 1))
    _check(_keys(_workload(batch, hq, hkv, table, lens, d), kind), scan)


@pytest.mark.parametrize("batch,hq,hkv,table,longest", [
    (2, 16, 2, 1024, 9003),     # eight heads
    (4, 32, 8, 2048, 32001),    # four, a wave of 128 units
])
@pytest.mark.parametrize("run,iters", [(run_entropic, 3), (run_fw, 3)])
def test_solves_with_a_block_to_an_sm(batch, hq, hkv, table, longest, run, iters):
    w = _workload(batch, hq, hkv, table, (longest,) + (513, 4100, 77)[: batch - 1])
    assert B.vsa_step_scan(B.shape_of(w.q, w.k_cache, w.block_table), 24, 100, B.VSA_STEP_SOLVE) == B.VSA_STEP_SCAN_INSIDE_MMA
    step, apart = run(w, iters, fused=True), run(w, iters)
    assert np.array_equal(step["routed"], apart["routed"]) and np.array_equal(step["fallback"], apart["fallback"])
    for name in apart["diag"]:
        if name != "lse":
            assert np.array_equal(step["diag"][name], apart["diag"][name], equal_nan=True), name
    assert np.array_equal(step["solve"], apart["solve"], equal_nan=True)
    units = batch * hq
    sparse = np.setdiff1d(np.arange(units), apart["fallback"])
    assert np.array_equal(step["out"].reshape(units, -1)[sparse], apart["out"].reshape(units, -1)[sparse])
