"""The dense pass with few groups, whose pages are spread over many blocks: odd and even numbers of items per group, fewer
items than warps, items of one page, one and all heads of a group listed."""
import math

import pytest

from gpu_runner import compare, run_gpu
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,d,page,lens,needles", [
    (1, 1, 128, 16, (4100,), 0),            # 17 items
    (3, 3, 64, 16, (5000, 257), 0),
    (8, 2, 64, 32, (8191, 300, 31), 0),
    (8, 1, 128, 16, (40001,), 0),           # one item per SM
    (8, 2, 256, 16, (2100, 97), 0),
    (16, 1, 128, 16, (3000,), 0),
    (8, 2, 128, 16, (6000, 6000, 6000), 3),
])
def test_items(hq, hkv, d, page, lens, needles):
    w = make_workload(WorkloadSpec(name="items", config=9, batch=len(lens), n_q_heads=hq, n_kv_heads=hkv, head_dim=d, P=2, K_c=16,
                                   seq_lens=lens, needles=needles, page_size=page), seed=8600 + hq + d + lens[0])
    for tau in (None, math.inf):
        compare(w, run_gpu(w) if tau is None else run_gpu(w, gap_threshold=tau), gap_threshold=tau)
