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


def clean_workload(batch, hq, hkv, P=32, K_c=100, d=128):
    # sequences 0 - 3 are the ones `poison` spoils; 2 has fewer pages than are routed, 1 and 3 have more
    lens = (2003, 1500, 100, 9001) + tuple(40 + 61 * (i % 19) for i in range(batch - 4))
    return make_workload(WorkloadSpec(name="nonfinite", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, P=P, K_c=K_c,
                                      seq_lens=lens, needles=1, head_dim=d), seed=4100 + batch)


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
