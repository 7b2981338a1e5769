"""The page scan over a list of pages (ragged batches in a pool that could not hold that many long sequences): parts that
cross sequences, single pages, ranges past the last page, groups of 1 to 16 heads, 32-token pages.  (Two heads a group
take the grid scan on the same kind of batch.)"""
import pytest

from gpu_runner import compare, run_gpu
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,page,long,short", [
    (8, 8, 16, 40000, (1, 16, 17, 127, 129, 2049)),
    (8, 4, 16, 33000, (5, 128, 1000, 4100)),
    (16, 4, 16, 30001, (2, 130, 700)),
    (16, 2, 32, 61000, (31, 33, 257, 5000)),
    (16, 1, 16, 60001, (90, 2100)),
])
def test_list_scan(hq, hkv, page, long, short):
    heads = hq // min(8, hq // hkv)     # KV heads as the scan sees them
    blocks = -(-(-(-long // page)) // 32)
    batch = 2 * 2368 // (heads * blocks) + 4      # more than two waves of warps
    lens = [short[i % len(short)] for i in range(batch)]
    lens[batch // 2] = long
    used = sum(-(-t // page) for t in lens)
    w = make_workload(WorkloadSpec(name="list", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, P=8, K_c=40,
                                   seq_lens=tuple(lens), needles=3, page_size=page, pool_pages=used + 5), seed=8100 + hq + hkv)
    assert w.block_table.shape[0] * w.block_table.shape[1] >= 2 * w.pool_pages
    assert batch * heads * blocks > 2 * 2368
    compare(w, run_gpu(w), dense_sample=4)

@pytest.mark.parametrize("hq,hkv,batch,blocks", [(16, 2, 28, 65), (8, 8, 19, 65)])
def test_list_scan_of_a_full_pool(hq, hkv, batch, blocks):
    # (sequences of one table width in a pool that holds them, from so many waves of warps on)
    assert 2 * batch * hkv * blocks >= (3 if hq > hkv else 8) * 2368
    pages = 32 * blocks - 5      # 2048 at least
    lens = [(1, 17, 300, 1025)[i % 4] for i in range(batch)]
    lens[0] = lens[-1] = pages * 16 - 3
    w = make_workload(WorkloadSpec(name="list", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, P=8, K_c=40,
                                   seq_lens=tuple(lens), needles=3, pool_pages=batch * pages // 2 + 1), seed=8500 + hq + hkv)
    assert w.block_table.shape[0] * w.block_table.shape[1] < 2 * w.pool_pages
    compare(w, run_gpu(w), dense_sample=4)
