"""The fused pass where a fifth block per SM saves a wave of blocks (593 - 740 and 1185 - 1480 units), and beside those counts."""
import pytest

from gpu_runner import compare, run_gpu
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,hq,hkv,d,P,K_c,page", [
    (19, 32, 8, 64, 8, 40, 16),      # 608 units
    (37, 20, 20, 64, 16, 128, 16),   # 740: five blocks on every SM
    (19, 32, 8, 128, 32, 256, 16),
    (20, 37, 37, 128, 5, 33, 32),
    (46, 32, 4, 128, 7, 50, 16),     # 1472
    (21, 32, 8, 256, 8, 64, 16),
    (20, 32, 8, 256, 64, 512, 16),   # five do not fit
    (24, 31, 31, 64, 8, 40, 16),     # 744: no wave saved
])
def test_blocks_per_sm(batch, hq, hkv, d, P, K_c, page):
    lens = tuple(40 + (97 * i) % (3 * P * page // 2 + 200) for i in range(batch))
    w = make_workload(WorkloadSpec(name="blocks", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, head_dim=d, P=P, K_c=K_c,
                                   seq_lens=lens, needles=2, page_size=page), seed=8400 + batch + hq + d)
    compare(w, run_gpu(w), dense_sample=4)
