"""Equal scores in such numbers that the fused kernel's page list (512 entries) or the list of its cut bucket (256)
overflows and the exact fallbacks decide, in every thread-block shape; rows whose last 16-byte chunk is partial."""
import pytest

from gpu_runner import compare, run_gpu
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,hq,hkv,P,K_c", [
    (2, 4, 2, 33, 200),      # 8 units: 512 threads
    (2, 4, 2, 128, 1030),    # the same with several tiles per group of lanes
    (40, 4, 2, 70, 513),     # 160 units: 256 threads
    (80, 4, 4, 64, 600),     # 320 units: 128 threads
    (2, 4, 2, 5, 40),        # fewer pages than the block has warps
    (80, 4, 4, 3, 30),
])
@pytest.mark.parametrize("distinct", [1, 3])
def test_equal_scores(batch, hq, hkv, P, K_c, distinct):
    lens = (9003,) + tuple(40 + 129 * (i % 23) for i in range(batch - 1))
    w = make_workload(WorkloadSpec(name="ties", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, P=P, K_c=K_c,
                                   seq_lens=lens, needles=0), seed=7000 + P)
    # `distinct` different key pages, repeated over the whole pool: whole classes of equal scores
    for i in range(w.k_cache.shape[0]):
        w.k_cache[i] = w.k_cache[i % distinct]
    if distinct == 1:
        w.k_cache[:] = w.k_cache[:, :, :1]   # and every token of a page equal
    compare(w, run_gpu(w), dense_sample=4)
