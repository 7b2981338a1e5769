"""The step whose page scores come from the tensor cores, in a cluster of the sparse pass's blocks and in a scan ahead of it: the routed
pages are those of the separate calls, whose scan has the fixed order, bit for bit and in the same order, and so is everything
that follows from them - for ordinary keys, for pages whose scores are equal, and for scores that differ in their last bits."""
import numpy as np
import pytest
import torch

from gpu_runner import compare, run_gpu
from test_gpu_fp8 import compare as compare_fp8, run_fp8
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu

LENS = (9003, 1, 16, 17, 512, 513, 1025, 4100, 529, 255)


def _workload(batch, hq, hkv, table, d=128, page=16, P=24, K_c=120):
    lens = tuple(LENS[i % len(LENS)] for i in range(batch))
    w = make_workload(WorkloadSpec(name="mma", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, P=P, K_c=K_c,
                                   seq_lens=lens, needles=4, needle_positions="uniform", page_size=page), seed=9100 + batch + hq)
    w.block_table = torch.nn.functional.pad(w.block_table, (0, table - w.block_table.shape[1]), value=-1)
    return w


SHAPES = [
    # a cluster scores the pages of its heads
    (1, 16, 2, 1040, 128, 16, 24),    # eight heads, 512 threads
    (10, 16, 2, 600, 128, 16, 24),    # 160 units of 256 threads
    (12, 16, 1, 600, 128, 16, 100),   # sixteen heads of one KV head
    (38, 4, 1, 2040, 128, 16, 24),    # four heads, two blocks to an SM
    (10, 16, 4, 2040, 64, 16, 24),
    (38, 4, 1, 2040, 256, 16, 24),
    (19, 8, 4, 2040, 128, 32, 24),    # two heads, pages of 32 tokens
    # scanned ahead
    (38, 8, 1, 1024, 128, 16, 24),
    (76, 4, 2, 1024, 128, 16, 3),     # two heads, fewer pages than warps
    (20, 16, 1, 1030, 128, 16, 64),
    (20, 16, 4, 4100, 128, 16, 24),   # four heads, long table
    (20, 16, 16, 1024, 64, 32, 24),   # one head
    (70, 16, 4, 1200, 64, 16, 24),    # 1120 units: five blocks to an SM
]


def _keys(w, kind):
    """Keys of every page: as generated; a few different pages only; one page with single elements moved by an ulp."""
    first = int(w.block_table[0, 0])            # (a page that a sequence has)
    if kind == "equal":
        some = w.k_cache[w.block_table[0, :3].long()].clone()
        for i in range(w.k_cache.shape[0]):
            w.k_cache[i] = some[i % 3]
    elif kind == "near":
        gen = torch.Generator().manual_seed(5)
        pool, hkv, page, d = w.k_cache.shape
        one = w.k_cache[first, :1, :1].clone().expand(pool, hkv, page, d).clone()
        at = torch.randint(0, d, (pool, hkv, 1, 1), generator=gen).expand(pool, hkv, page, 1)
        up = torch.randint(-1, 2, (pool, hkv, 1, 1), generator=gen, dtype=torch.int16).expand(pool, hkv, page, 1)
        bits = one.view(torch.int16)
        bits.scatter_(3, at, bits.gather(3, at) + up)
        w.k_cache = one
    return w


@pytest.mark.parametrize("kind", ["generated", "equal", "near"])
@pytest.mark.parametrize("batch,hq,hkv,table,d,page,P", SHAPES)
def test_step(batch, hq, hkv, table, d, page, P, kind):
    w = _keys(_workload(batch, hq, hkv, table, d, page, P, min(120, P * page // 2)), kind)
    g = run_gpu(w)
    assert np.array_equal(g.step_routed, g.routed_pages)
    for name in g.step_diag:
        if name != "lse":                       # (rewritten by the dense pass where a unit falls back)
            assert np.array_equal(g.step_diag[name], g.diag[name], equal_nan=True), name
    assert np.array_equal(g.step_fallback_units, g.fallback_units)
    sparse = np.setdiff1d(np.arange(batch * hq), g.fallback_units)
    assert np.array_equal(g.step_out.reshape(batch * hq, -1)[sparse], g.out.reshape(batch * hq, -1)[sparse])


@pytest.mark.parametrize("shape", [SHAPES[0], SHAPES[7]])
def test_against_the_oracle(shape):
    w = _workload(*shape, 100)
    compare(w, run_gpu(w), dense_sample=2)


def test_pages_outside_the_pool():
    """Entries that name no page score -inf: the last in the order, by position; a unit that routes one fails."""
    for batch, hq, hkv, table in ((10, 16, 2, 600), (38, 8, 1, 1024)):
        w = _workload(batch, hq, hkv, table)
        ref = run_gpu(w)
        w.block_table[0, 5:500:3] = w.k_cache.shape[0] + 9
        w.block_table[4, 2:30] = -1
        got = run_gpu(w, summaries=ref.summaries)
        assert np.array_equal(got.step_routed, got.routed_pages)
        assert np.array_equal(got.step_diag["status"], got.diag["status"]) and got.diag["status"].reshape(batch, hq)[4].all()


def test_fp8():
    compare_fp8(*run_fp8(_workload(10, 16, 2, 600)))
    compare_fp8(*run_fp8(_workload(38, 8, 1, 1024)))


@pytest.mark.parametrize("kind", ["entropic", "frank_wolfe"])
def test_solvers(kind):
    """256 threads, one block to an SM and two."""
    from paper_2602_13804_b200 import binding as B
    for batch, hq, hkv in ((2, 16, 2), (10, 16, 2)):
        w = _workload(batch, hq, hkv, 1040, K_c=100)
        g = run_gpu(w)
        wd = w.to("cuda:0")
        shape, units = B.shape_of(wd.q, wd.k_cache, wd.block_table), batch * hq
        out, diag, sol = torch.empty_like(wd.q, dtype=torch.float32), B.alloc_diag(units, "cuda:0"), B.alloc_solve(units, "cuda:0")
        routed = torch.empty((batch, hq, 24), dtype=torch.int32, device="cuda:0")
        flist, fcount = torch.empty(units, dtype=torch.int32, device="cuda:0"), torch.zeros(1, dtype=torch.int32, device="cuda:0")
        getattr(B, "vsa_decode_step_" + kind)(shape, wd.q, g.summaries, wd.k_cache, wd.v_cache, wd.block_table, wd.seq_lens, 24, 100,
                                              w.epsilon, w.gap_threshold, 3, out, diag, sol, routed, flist, fcount,
                                              B.alloc_workspace(shape, 24, 100, B.VSA_WS_STEP, "cuda:0"))
        torch.cuda.synchronize()
        assert np.array_equal(routed.cpu().numpy(), g.routed_pages)


@pytest.mark.parametrize("d", [64, 128])
def test_rounding_stays_within_the_slack(d):
    """The scores that the scan leaves in the workspace, against fp64: half of the slack is 40 * 2^-23 * A for a score
    and the fixed order together, of which the latter needs 5 at most.  Magnitudes spread over 2^16, with cancellation."""
    from paper_2602_13804_b200 import binding as B
    w = _workload(38, 8, 1, 1024, d)
    gen = torch.Generator().manual_seed(d)
    spread = torch.exp2(torch.randint(-8, 9, (1, 1, 1, d), generator=gen).float())
    w.k_cache = (w.k_cache.float() * spread * torch.exp2(torch.randint(-3, 4, (w.k_cache.shape[0], 1, 1, 1), generator=gen).float())).bfloat16()
    wd = w.to("cuda:0")
    shape, units, P = B.shape_of(wd.q, wd.k_cache, wd.block_table), 38 * 8, 24
    summ = torch.zeros((shape.num_pool_pages, 1, d), dtype=torch.bfloat16, device="cuda:0")
    B.vsa_build_page_summaries(shape, wd.k_cache, wd.block_table, wd.seq_lens, None, summ)
    ws = B.alloc_workspace(shape, P, 100, B.VSA_WS_STEP, "cuda:0")
    B.vsa_decode_step(shape, wd.q, summ, wd.k_cache, wd.v_cache, wd.block_table, wd.seq_lens, P, 100, w.epsilon, w.gap_threshold,
                      torch.empty((38, 8, d), device="cuda:0"), B.alloc_diag(units, "cuda:0"),
                      torch.empty((38, 8, P), dtype=torch.int32, device="cuda:0"), torch.empty(units, dtype=torch.int32, device="cuda:0"),
                      torch.zeros(1, dtype=torch.int32, device="cuda:0"), ws)
    torch.cuda.synchronize()
    got = ws.view(torch.uint8)[: units * 1024 * 4].view(torch.float32).view(38, 8, 1024).double()
    worst = 0.0
    for b in (0, 7, 8):
        n = -(-int(w.seq_lens[b]) // 16)
        rows = summ[wd.block_table[b, :n].long(), 0].double()
        want, a = wd.q[b].double() @ rows.T, wd.q[b].double().abs() @ rows.abs().T
        worst = max(worst, float(((got[b, :, :n] - want).abs() / a).max()) * 2.0 ** 23)
    print("largest rounding error in units of 2^-23 A:", worst)
    assert worst <= 35.0
