"""The dense pass over an e4m3 cache brings whole tiles of 16 rows: lengths around one and two tiles and around the warps'
rounds, with NaN bytes in every row that belongs to no sequence (rows past a length, pages of no table)."""
import math

import pytest
import torch

from gpu_runner import compare
from test_gpu_fp8 import run_fp8, spec
from workloads import make_workload, quantize_kv_fp8

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("page,hq,hkv,lens,alt", [
    (16, 8, 2, (9, 15, 16, 17, 31, 32, 33, 47), False),
    (16, 4, 4, (383, 384, 385, 767, 769, 10), False),        # twelve warps, 32 tokens each
    (16, 16, 2, (13000, 12289, 100), True),                  # more than 32 units of a warp's look-up in one item
    (32, 8, 2, (9, 16, 17, 33, 49, 64, 65, 1000), False),
    (32, 16, 1, (2049, 31), True),
])
def test_rows_outside_the_sequences(page, hq, hkv, lens, alt):
    w = make_workload(spec(batch=len(lens), n_q_heads=hq, n_kv_heads=hkv, seq_lens=lens, page_size=page, P=2, K_c=8, needles=1),
                      seed=8300 + page + hq + lens[0])
    wq, k8, v8, ke, ve = quantize_kv_fp8(w)
    outside = torch.ones((k8.shape[0], page), dtype=torch.bool)
    for b, T in enumerate(lens):
        for i in range(-(-T // page)):
            outside[int(w.block_table[b, i]), :min(page, T - i * page)] = False
    at = outside[:, None, :].expand(-1, hkv, -1)
    k8[at], v8[at] = 0x7f, 0xff
    wq, g = run_fp8(w, gap_threshold=math.inf, alt_strides=alt, quantised=(wq, k8, v8, ke, ve))
    compare(wq, g, gap_threshold=math.inf)


@pytest.mark.parametrize("page,token,head_pad,page_pad", [(16, 144, 32, 48), (32, 128, 16, 0), (16, 272, 0, 4096)])
def test_padded_strides(page, token, head_pad, page_pad):
    lens, hkv = (700, 33, 16), 2
    w = make_workload(spec(batch=len(lens), n_q_heads=8, n_kv_heads=hkv, seq_lens=lens, page_size=page, P=2, K_c=8), seed=8400 + page + token)
    wq, k8, v8, ke, ve = quantize_kv_fp8(w)
    head = page * token + head_pad
    strides = (hkv * head + page_pad, head, token, 1)

    def padded(x):
        out = torch.full((x.shape[0] * strides[0],), 0x7f, dtype=torch.uint8, device="cuda:0").as_strided(x.shape, strides)
        out.copy_(x)
        return out

    wq, g = run_fp8(w, gap_threshold=math.inf, quantised=(wq, padded(k8), padded(v8), ke, ve))
    compare(wq, g, gap_threshold=math.inf)
