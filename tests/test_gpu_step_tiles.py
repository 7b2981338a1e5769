"""The fused sparse pass where its tiles and batches end: several rounds of key tiles in every thread-block size (bulk copies
in blocks of 128 threads, row by row where the rows are not contiguous), candidate counts beside the value gather's batches,
score rows of one chunk per thread and of one chunk more."""
import pytest

from gpu_runner import compare, run_gpu
from test_gpu_fp8 import compare as _compare, run_fp8
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu


def _workload(batch, hq, hkv, P, K_c, lens, **kw):
    return make_workload(WorkloadSpec(name="tiles", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, P=P, K_c=K_c,
                                      seq_lens=lens, needles=2, needle_positions="uniform", **kw), seed=8000 + P + K_c)


def _strided(w):
    wd = w.to("cuda:0")
    wd.k_cache = wd.k_cache.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    wd.v_cache = wd.v_cache.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)
    return wd


@pytest.mark.parametrize("batch,P,K_c,d,page", [
    (40, 9, 33, 128, 16),     # 320 units: 128 threads, two rounds, the second with one tile
    (40, 64, 481, 128, 32),   # sixteen rounds
    (40, 40, 65, 64, 16),
    (40, 21, 255, 256, 16),
    (20, 33, 63, 128, 16),    # 160 units: 256 threads
    (20, 40, 129, 64, 32),
    (2, 33, 97, 128, 16),     # 16 units: 512 threads
])
@pytest.mark.parametrize("native", [True, False])
def test_tiles_and_batches(batch, P, K_c, d, page, native):
    lens = tuple(37 + 61 * (i % 17) for i in range(batch - 1)) + (2900,)
    w = _workload(batch, 8, 2, P, K_c, lens, head_dim=d, page_size=page)
    compare(w, run_gpu(w if native else _strided(w)), dense_sample=4)


@pytest.mark.parametrize("alt", [False, True])
def test_fp8_tiles(alt):
    w = _workload(40, 8, 2, 25, 65, tuple(37 + 61 * (i % 17) for i in range(40)))
    _compare(*run_fp8(w, alt_strides=alt))


@pytest.mark.parametrize("batch,threads", [(2, 512), (20, 256), (40, 128)])
@pytest.mark.parametrize("over", [-3, 0, 1, 4, 9])
def test_one_chunk_per_thread(batch, threads, over):
    pages = 4 * threads + over   # (a score row starts at any word of its first 16-byte chunk)
    w = _workload(batch, 8, 2, 7, 30, (16 * pages - 5,) + tuple(16 * (3 + i) for i in range(batch - 1)))
    compare(w, run_gpu(w), dense_sample=2)
