"""The dense pass over an e4m3 cache whose value scales lie far apart within one sequence.  Tokens of large values have keys
opposite to the group's query (scores lower by about 4 |q|^2 / sqrt(d) = 45, weights below 2^-60), so the result is that of
the small pages alone: a page's share must not lose bits to the scale of a page met before it, or of the other page of a
32-token unit.  2^40 * 2^-60 * max|v| is far below the tolerances of gpu_runner, which hold as they are."""
import math

import pytest
import torch

from gpu_runner import compare
from paper_2602_13804_b200 import binding as B
from test_gpu_fp8 import run_fp8, spec
from workloads import make_workload, quantize_kv_fp8

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

WARP_ROUND = 12 * 32    # tokens that the twelve warps of a block take before a warp's second unit


@pytest.mark.parametrize("page,run,lens", [
    (16, WARP_ROUND, (4 * WARP_ROUND, 7 * WARP_ROUND + 5)),   # every warp meets large pages first
    (32, WARP_ROUND, (4 * WARP_ROUND, 7 * WARP_ROUND + 5)),
    (16, 16, (1000, 333)),                                    # large and small pages in turn, both in every unit
])
@pytest.mark.parametrize("octaves", [20, 40])
def test_large_pages_without_weight(page, run, lens, octaves):
    hq, hkv, G = 8, 2, 4
    w = make_workload(spec(batch=len(lens), n_q_heads=hq, n_kv_heads=hkv, seq_lens=lens, page_size=page, P=2, K_c=8, needles=0),
                      seed=8700 + page + run + octaves)
    w.q[:] = w.q[:, ::G].repeat_interleave(G, dim=1)          # one direction per group, so that its heads agree
    for b, T in enumerate(lens):
        for t in range(T):
            if (t // run) % 2 == 0:
                phys, row = int(w.block_table[b, t // page]), t % page
                w.k_cache[phys, :, row] = -4 * w.q[b, ::G]
                w.v_cache[phys, :, row] *= 2.0 ** octaves
    wq, g = run_fp8(w, gap_threshold=math.inf, quantised=quantize_kv_fp8(w))
    stats = compare(wq, g, gap_threshold=math.inf)
    assert stats["fallback_fraction"] == 1.0


def test_scales_of_either_sign():
    """value = e4m3(byte) * scale: a negative scale with the bytes' signs turned is the same cache, bit for bit."""
    w = make_workload(spec(seq_lens=(700, 333, 45), needles=0), seed=8790)
    _, k8, v8, ke, ve = quantize_kv_fp8(w)
    odd = (torch.arange(ve.numel()) % 2 == 1).view(ve.shape)
    q, bt, sl, k8, ks = (x.to(DEV) for x in (w.q, w.block_table, w.seq_lens, k8, torch.exp2(ke.float())))
    shape = B.shape_of(q, k8, bt)
    ws = B.alloc_workspace(shape, w.spec.P, w.spec.K_c, B.VSA_WS_DENSE, DEV)

    def dense(v8, vs):
        out = torch.full((shape.batch, shape.n_q_heads, 128), float("nan"), dtype=torch.float32, device=DEV)
        B.vsa_dense_decode_fallback_fp8(shape, q, k8, v8.to(DEV), ks, vs.to(DEV), bt, sl, None, None, w.epsilon, out, None, ws)
        return out.cpu()

    scale = torch.exp2(ve.float())
    plain = dense(v8, scale)
    turned = dense(torch.where(odd[:, :, None, None], v8 ^ 0x80, v8), torch.where(odd, -scale, scale))
    assert torch.isfinite(plain).all() and plain.abs().max() > 0.1
    assert torch.equal(plain, turned)
