"""NaN and infinity in the queries and in cached keys.  Their results are not specified, but a step that meets them
stays inside its buffers: every routed page lies inside the sequence, and the other sequences of the batch get bit for
bit what they get without them (and that is what the oracle says)."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from gpu_runner import compare, run_gpu
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu
NAN, INF = float("nan"), float("inf")


def clean_workload(batch, hq, hkv, P=32, K_c=100, d=128, table=0):
    # sequences 0 - 3 are the ones `poison` spoils; 2 has fewer pages than are routed, 1 and 3 have more
    lens = (2003, 1500, 100, 9001) + tuple(40 + 61 * (i % 19) for i in range(batch - 4))
    w = make_workload(WorkloadSpec(name="nonfinite", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, P=P, K_c=K_c,
                                   seq_lens=lens, needles=1, head_dim=d), seed=4100 + batch)
    if table:                              # a wider block table, whose width decides where the pages are scored
        w.block_table = torch.nn.functional.pad(w.block_table, (0, table - w.block_table.shape[1]), value=-1)
    return w


def shape_of(w):
    from paper_2602_13804_b200 import binding as B
    return B.shape_of(w.q, w.k_cache, w.block_table)


def poison(w):
    """A copy of w with non-finite values in sequences 0 - 3."""
    q, k = w.q.clone(), w.k_cache.clone()
    q[0, 0, 5] = NAN                       # every score is NaN
    q[0, 1, 3], q[0, 1, 9] = INF, -INF     # NaN or +-inf
    q[0, 2, :] = -3.3e38                   # sums that overflow
    q[0, 3, :] = 0.0
    q[0, 3, 1] = -INF                      # +inf, -inf, and NaN where the key is 0
    bt = w.block_table
    k[bt[1, 40], 0, 3, 7] = NAN            # one key of a long sequence
    k[bt[2, 1], 0, 0, 0] = NAN             # one key of a sequence with fewer pages than are routed
    k[bt[2, 4], -1, 2, 0] = -INF
    pages = bt[3, : -(-int(w.seq_lens[3]) // w.spec.page_size)].long()
    k[pages[5:], 0] = NAN                  # nearly every key of a long sequence
    return replace(w, q=q, k_cache=k)


def check_pages(routed, w, P):
    """Every unit's list: min(P, pages) distinct pages of the sequence, then -1."""
    for b in range(w.spec.batch):
        nb = -(-int(w.seq_lens[b]) // w.spec.page_size)
        n = min(P, nb)
        r = routed[b].reshape(-1, P)
        assert (r[:, :n] >= 0).all() and (r[:, :n] < nb).all() and (r[:, n:] == -1).all(), f"sequence {b}"
        assert all(len(set(row[:n].tolist())) == n for row in r), f"sequence {b}"


@pytest.mark.parametrize("batch,hq,hkv,P,K_c,d", [
    (6, 8, 2, 32, 100, 128),      # 48 units: 512 threads
    (6, 8, 8, 128, 2048, 128),    # more pages and candidates than any unit but one has
    (20, 8, 4, 32, 300, 128),     # 160 units: 256 threads
    (40, 8, 2, 64, 100, 128),     # 320 units: 128 threads
    (224, 8, 1, 32, 100, 128),    # 1792 units: five blocks of 128 threads per SM
    (6, 8, 2, 32, 100, 64),
    (40, 8, 2, 32, 100, 64),
    (6, 8, 2, 32, 100, 256),
    (20, 8, 4, 32, 300, 256),
])
def test_step(batch, hq, hkv, P, K_c, d):
    w = clean_workload(batch, hq, hkv, P, K_c, d)
    ref = run_gpu(w, gap_threshold=-INF)
    compare(w, ref, gap_threshold=-INF)
    got = run_gpu(poison(w), gap_threshold=-INF)
    check_pages(got.step_routed, w, P)
    check_pages(got.routed_pages, w, P)
    assert np.array_equal(got.step_routed, got.routed_pages)     # one order everywhere: NaN first, then by score
    for name in ("out", "step_out", "step_routed"):
        assert np.array_equal(getattr(got, name)[4:], getattr(ref, name)[4:]), name
    for name in ref.step_diag:
        assert np.array_equal(got.step_diag[name][4 * hq:], ref.step_diag[name][4 * hq:]), name
    # the page that holds the NaN key has a NaN score, which ranks first for every head that reads it
    assert (got.step_routed[1, : hq // hkv, 0] == 40).all()


@pytest.mark.parametrize("batch,hq,hkv,P,K_c,d,table,scan", [
    (6, 16, 2, 32, 100, 128, 563, "INSIDE"),           # 512 threads, more rounds than one
    (5, 4, 1, 32, 100, 64, 563, "INSIDE"),             # with helpers
    (13, 8, 2, 32, 100, 128, 4096, "INSIDE_MMA"),      # 512 threads
    (10, 16, 2, 32, 100, 128, 600, "INSIDE_MMA"),      # 256, eight heads
    (20, 8, 2, 64, 300, 128, 2048, "INSIDE_MMA"),
    (10, 16, 4, 32, 100, 64, 2040, "INSIDE_MMA"),
    (38, 4, 1, 32, 300, 256, 2040, "INSIDE_MMA"),
    (40, 8, 1, 64, 100, 128, 1024, "AHEAD_MMA"),       # 128 threads
    (150, 8, 1, 32, 100, 64, 1024, "AHEAD_MMA"),       # five blocks of 128 threads per SM
])
def test_scans(batch, hq, hkv, P, K_c, d, table, scan):
    """Every place where a step scores the pages.  Beside the values of `poison`: products that overflow where a sum in another order need
    not, and sums of such size that cancel, whose pages rank among ordinary ones."""
    from paper_2602_13804_b200 import binding as B
    w = clean_workload(batch, hq, hkv, P, K_c, d, table)
    assert B.vsa_step_scan(shape_of(w), P, K_c) == getattr(B, "VSA_STEP_SCAN_" + scan)
    ref = run_gpu(w, gap_threshold=-INF)
    bad = poison(w)
    bt = bad.block_table
    bad.q[1, 0, 20:24] = torch.tensor([3e19, 3e19, 2.0, 0.0], dtype=torch.bfloat16)
    for page, tail in ((3, 1.0), (7, 30.0), (11, -5.0), (60, 1e4)):      # 9e38 - 9e38 (an overflow: NaN or an infinity) + ...
        bad.k_cache[bt[1, page], 0, :, 20:23] = torch.tensor([3e19, -3e19, tail], dtype=torch.bfloat16)
    for page, tail in ((4, 1.0), (9, 30.0), (44, 300.0)):                # 9e37 - 9e37 + ...
        bad.k_cache[bt[1, page], 0, :, 20:23] = torch.tensor([3e18, -3e18, tail], dtype=torch.bfloat16)
    got = run_gpu(bad, gap_threshold=-INF)
    check_pages(got.step_routed, w, P)
    check_pages(got.routed_pages, w, P)
    assert np.array_equal(got.step_routed, got.routed_pages)
    for name in ("out", "step_out", "step_routed"):
        assert np.array_equal(getattr(got, name)[4:], getattr(ref, name)[4:]), name
    for name in ref.step_diag:
        assert np.array_equal(got.step_diag[name][4 * hq:], ref.step_diag[name][4 * hq:]), name
        assert np.array_equal(got.step_diag[name], got.diag[name], equal_nan=True), name
    assert (got.step_routed[1, 1 : hq // hkv, 0] == 40).all()


@pytest.mark.parametrize("batch,hq,hkv,P,table,scan", [
    (20, 8, 2, 32, 2048, "INSIDE_MMA"), (13, 8, 2, 32, 4096, "INSIDE_MMA"), (40, 8, 1, 64, 1024, "AHEAD_MMA"), (6, 16, 2, 32, 563, "INSIDE"),
])
def test_one_nan_key_costs_little(batch, hq, hkv, P, table, scan):
    """One NaN in every sequence: only the pages that it spoils are scored anew.  (Scoring every page anew took more than twice the
    time of the step; 1.6 leaves room for the clock of a shared machine.)"""
    from paper_2602_13804_b200 import SparsePagedDecoder
    from paper_2602_13804_b200 import binding as B
    T, dev = table * 16, "cuda:0"
    gen = torch.Generator(device=dev).manual_seed(3)
    shape = B.make_shape(batch, hq, hkv, table, table)                   # (all sequences share their pages)
    assert B.vsa_step_scan(shape, P, 100) == getattr(B, "VSA_STEP_SCAN_" + scan)
    k = torch.randn((table, hkv, 16, 128), generator=gen, device=dev).bfloat16()
    bt = torch.arange(table, dtype=torch.int32, device=dev).expand(batch, -1).contiguous()
    lens = torch.full((batch,), T, dtype=torch.int32, device=dev)
    q = torch.randn((batch, hq, 128), generator=gen, device=dev).bfloat16()
    dec = SparsePagedDecoder(shape, P, 100, 11.0, -INF, device=dev)
    us = []
    for spoil in (False, True):
        if spoil:
            k[5, :, 0, 0] = NAN
        summ = dec.build_summaries(k, bt, lens)
        best = INF
        for _ in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                dec.step(q, summ, k, k, bt, lens)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 50.0)
        us.append(best)
    assert us[1] < 1.6 * us[0], us


@pytest.mark.parametrize("batch,hq,hkv,P", [(6, 8, 2, 32), (40, 8, 2, 64)])
def test_step_fp8(batch, hq, hkv, P):
    """The e4m3 cache: NaN bytes in the same places, non-finite queries."""
    from paper_2602_13804_b200 import binding as B
    from workloads import quantize_kv_fp8
    dev = "cuda:0"
    w, k8, v8, ke, ve = quantize_kv_fp8(clean_workload(batch, hq, hkv, P))
    bad = poison(w)
    k8_bad = k8.clone()
    k8_bad.view(torch.uint8)[torch.isnan(bad.k_cache)] = 0x7f
    wd = w.to(dev)
    shape = B.shape_of(wd.q, k8.to(dev), wd.block_table)
    units = batch * hq
    ks, vs, v8 = torch.exp2(ke.float()).to(dev), torch.exp2(ve.float()).to(dev), v8.to(dev)

    def run(q, k8):
        summ = torch.zeros((shape.num_pool_pages, hkv, 128), dtype=torch.bfloat16, device=dev)
        B.vsa_build_page_summaries_fp8(shape, k8, ks, wd.block_table, wd.seq_lens, None, summ)
        out = torch.empty((batch, hq, 128), dtype=torch.float32, device=dev)
        diag, flist = B.alloc_diag(units, dev), torch.empty(units, dtype=torch.int32, device=dev)
        routed, fcount = torch.empty((batch, hq, P), dtype=torch.int32, device=dev), torch.zeros(1, dtype=torch.int32, device=dev)
        B.vsa_decode_step_fp8(shape, q, summ, k8, v8, ks, vs, wd.block_table, wd.seq_lens, P, 100, w.epsilon, -INF, out,
                              diag, routed, flist, fcount, B.alloc_workspace(shape, P, 100, B.VSA_WS_STEP, dev))
        torch.cuda.synchronize()
        return out.cpu(), diag.cpu(), routed.cpu()

    out, diag, routed = run(wd.q, k8.to(dev))
    out_b, diag_b, routed_b = run(bad.q.to(dev), k8_bad.to(dev))
    check_pages(routed_b.numpy(), w, P)
    assert torch.equal(out_b[4:], out[4:]) and torch.equal(routed_b[4:], routed[4:])
    assert torch.equal(diag_b[4 * hq:], diag[4 * hq:])


@pytest.mark.parametrize("batch,K_c", [(6, 32), (6, 250), (40, 32)])
@pytest.mark.parametrize("method", ["entropic", "frank_wolfe"])
def test_solvers(method, batch, K_c):
    """Iterative weights: the vertex that Frank-Wolfe picks is a candidate whatever the gradients are."""
    from paper_2602_13804_b200 import binding as B
    dev, hq, hkv, P = "cuda:0", 8, 2, 32
    w = clean_workload(batch, hq, hkv, P, K_c)

    def run(w):
        wd = w.to(dev)
        shape = B.shape_of(wd.q, wd.k_cache, wd.block_table)
        units = batch * hq
        summ = torch.zeros((shape.num_pool_pages, hkv, 128), dtype=torch.bfloat16, device=dev)
        B.vsa_build_page_summaries(shape, wd.k_cache, wd.block_table, wd.seq_lens, None, summ)
        out = torch.empty((batch, hq, 128), dtype=torch.float32, device=dev)
        diag, sol, flist = B.alloc_diag(units, dev), B.alloc_solve(units, dev), torch.empty(units, dtype=torch.int32, device=dev)
        routed, fcount = torch.empty((batch, hq, P), dtype=torch.int32, device=dev), torch.zeros(1, dtype=torch.int32, device=dev)
        getattr(B, "vsa_decode_step_" + method)(shape, wd.q, summ, wd.k_cache, wd.v_cache, wd.block_table, wd.seq_lens, P, K_c,
                                                w.epsilon, -INF, 4, out, diag, sol, routed, flist, fcount,
                                                B.alloc_workspace(shape, P, K_c, B.VSA_WS_STEP, dev))
        torch.cuda.synchronize()
        return out.cpu(), diag.cpu(), sol.cpu(), routed.cpu()

    out, diag, sol, routed = run(w)
    out_b, diag_b, sol_b, routed_b = run(poison(w))
    check_pages(routed_b.numpy(), w, P)
    assert torch.equal(out_b[4:], out[4:]) and torch.equal(routed_b[4:], routed[4:])
    assert torch.equal(diag_b[4 * hq:], diag[4 * hq:]) and torch.equal(sol_b[4 * hq:], sol[4 * hq:])


@pytest.mark.parametrize("variant", ["certified", "expand", "two_level", "group_shared"])
@pytest.mark.parametrize("batch", [6, 40])
def test_routing_variants(variant, batch):
    from paper_2602_13804_b200 import binding as B
    dev, hq, hkv, P, K_c = "cuda:0", 8, 2, 32, 100
    w = clean_workload(batch, hq, hkv, P, K_c)

    def run(w):
        wd = w.to(dev)
        shape = B.shape_of(wd.q, wd.k_cache, wd.block_table)
        units = batch * hq
        summ = torch.zeros((shape.num_pool_pages, hkv, 128), dtype=torch.bfloat16, device=dev)
        B.vsa_build_page_summaries(shape, wd.k_cache, wd.block_table, wd.seq_lens, None, summ)
        out = torch.empty((batch, hq, 128), dtype=torch.float32, device=dev)
        diag, flist = B.alloc_diag(units, dev), torch.empty(units, dtype=torch.int32, device=dev)
        fcount, cert = torch.zeros(1, dtype=torch.int32, device=dev), B.alloc_cert(units, dev)
        radii = torch.zeros((shape.num_pool_pages, hkv), dtype=torch.float32, device=dev)
        B.vsa_build_page_radii(shape, wd.k_cache, summ, wd.block_table, wd.seq_lens, None, radii)
        routed = torch.empty((batch, hkv if variant == "group_shared" else hq, 64 if variant == "expand" else P),
                             dtype=torch.int32, device=dev)
        cache = (wd.k_cache, wd.v_cache, wd.block_table, wd.seq_lens)
        after = (K_c, w.epsilon, -INF, out, diag)
        if variant == "two_level":
            sup = torch.zeros((batch, B.n_super_pages(shape), hkv, 128), dtype=torch.bfloat16, device=dev)
            B.vsa_build_super_summaries(shape, summ, wd.block_table, wd.seq_lens, None, sup)
            B.vsa_decode_step_two_level(shape, wd.q, summ, sup, *cache, 4, P, *after, routed, flist, fcount,
                                        B.alloc_workspace(shape, 4, K_c, B.VSA_WS_STEP_TWO_LEVEL, dev))
        elif variant == "group_shared":
            B.vsa_decode_step_group_shared(shape, wd.q, summ, *cache, P, *after, routed, flist, fcount,
                                           B.alloc_workspace(shape, P, K_c, B.VSA_WS_STEP, dev))
        elif variant == "expand":
            B.vsa_decode_step_certified_expand(shape, wd.q, summ, radii, *cache, P, 64, *after, cert, routed, flist, fcount,
                                               B.alloc_workspace(shape, 64, K_c, B.VSA_WS_STEP_EXPAND, dev))
        else:
            B.vsa_decode_step_certified(shape, wd.q, summ, radii, *cache, P, *after, cert, routed, flist, fcount,
                                        B.alloc_workspace(shape, P, K_c, B.VSA_WS_STEP_CERTIFIED, dev))
        torch.cuda.synchronize()
        return out.cpu(), diag.cpu(), routed.cpu().numpy()

    out, diag, routed = run(w)
    out_b, diag_b, routed_b = run(poison(w))
    for b in range(batch):
        nb = -(-int(w.seq_lens[b]) // w.spec.page_size)
        assert ((routed_b[b] >= -1) & (routed_b[b] < nb)).all()
        for row in routed_b[b]:
            row = row[row >= 0]
            assert len(set(row.tolist())) == len(row) > 0
    assert torch.equal(out_b[4:], out[4:]) and np.array_equal(routed_b[4:], routed[4:])
    assert torch.equal(diag_b[4 * hq:], diag[4 * hq:])
