"""The step with events between its kernels runs what the step runs: every result bit for bit the same, wherever the pages
are scored - ahead of the sparse pass or inside it, in the fixed order or by MMAs."""
import pytest
import torch

from paper_2602_13804_b200 import binding as B
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,hq,hkv,table,d,scan", [
    (1, 32, 8, 256, 128, B.VSA_STEP_SCAN_INSIDE),
    (4, 32, 8, 4096, 128, B.VSA_STEP_SCAN_INSIDE_MMA),     # 512 threads
    (8, 32, 8, 2048, 128, B.VSA_STEP_SCAN_INSIDE_MMA),     # 256
    (2, 32, 8, 2048, 128, B.VSA_STEP_SCAN_AHEAD),
    (38, 8, 1, 1024, 128, B.VSA_STEP_SCAN_AHEAD_MMA),
    (8, 32, 8, 2048, 64, B.VSA_STEP_SCAN_INSIDE_MMA),
])
def test_timed_step(batch, hq, hkv, table, d, scan):
    lens = tuple(max(1, 3001 - 317 * (b % 9)) for b in range(batch))
    w = make_workload(WorkloadSpec(name="timed", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, P=32, K_c=200, seq_lens=lens,
                                   needles=1, needle_positions="uniform"), seed=8200 + batch)
    w.block_table = torch.nn.functional.pad(w.block_table, (0, table - w.block_table.shape[1]), value=-1)
    wd = w.to("cuda:0")
    shape, units, P, K_c = B.shape_of(wd.q, wd.k_cache, wd.block_table), batch * hq, 32, 200
    assert B.vsa_step_scan(shape, P, K_c) == scan
    summ = torch.zeros((shape.num_pool_pages, hkv, d), dtype=torch.bfloat16, device="cuda:0")
    B.vsa_build_page_summaries(shape, wd.k_cache, wd.block_table, wd.seq_lens, None, summ)

    def run(*events):
        out = torch.full((batch, hq, d), float("nan"), device="cuda:0")
        diag, routed = B.alloc_diag(units, "cuda:0"), torch.empty((batch, hq, P), dtype=torch.int32, device="cuda:0")
        flist, fcount = torch.full((units,), -1, dtype=torch.int32, device="cuda:0"), torch.zeros(1, dtype=torch.int32, device="cuda:0")
        step = B.vsa_decode_step_timed if events else B.vsa_decode_step
        step(shape, wd.q, summ, wd.k_cache, wd.v_cache, wd.block_table, wd.seq_lens, P, K_c, w.epsilon, 4.0, out, diag, routed, flist,
             fcount, B.alloc_workspace(shape, P, K_c, B.VSA_WS_STEP, "cuda:0"), *events)
        torch.cuda.synchronize()
        return out, diag, routed, flist.sort().values, fcount

    events = [torch.cuda.Event(enable_timing=True) for _ in range(5)]
    for e in events:
        e.record()
    for a, b in zip(run(), run(events)):
        assert torch.equal(a, b)
    assert all(events[i].elapsed_time(events[i + 1]) >= 0.0 for i in range(4))
    assert events[2].elapsed_time(events[3]) > 0.0 and events[3].elapsed_time(events[4]) > 0.0
