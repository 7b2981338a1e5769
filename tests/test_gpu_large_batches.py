"""The scan ahead by MMAs with batches whose lengths several warps of a block sum up: results as from the separate calls, bit for
bit, and no slower than the fixed-order scan that a table of one page less takes."""
import torch
import pytest

from paper_2602_13804_b200 import SparsePagedDecoder
from paper_2602_13804_b200 import binding as B
from test_gpu_scan_rounds import _check, _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,hq,hkv", [(149, 2, 1), (256, 2, 1), (257, 2, 1), (600, 8, 1), (2048, 4, 2), (4096, 2, 1)])
def test_large_batches(batch, hq, hkv):
    """Lengths by the warps of a block, 32 at a time; sequences without a usable length among them, and the last ones."""
    lens = [1 + (977 * i) % 640 for i in range(batch)]
    w = _workload(batch, hq, hkv, 1024, lens, P=8, K_c=40)
    w.seq_lens[3::7] = 0
    w.seq_lens[-1] = -5
    w.seq_lens[batch // 2] = 1024 * 16 + 1
    _check(w, "AHEAD_MMA")


def test_many_short_sequences_cost_no_more():
    """2048 sequences of 64 to 16k tokens.  (One warp that sums the lengths alone takes 20 us of the step's 131, where the
    fixed order takes 113; 1.08 leaves room for the clock of a shared machine.)"""
    batch, P, dev = 2048, 16, "cuda:0"
    gen = torch.Generator(device=dev).manual_seed(3)
    lens = (64.0 * torch.exp2(8.0 * torch.arange(batch, device=dev) / batch)).int().clamp_(max=1023 * 16)
    k = torch.randn((1024, 1, 16, 128), generator=gen, device=dev).bfloat16()        # (all sequences share their pages)
    q = torch.randn((batch, 2, 128), generator=gen, device=dev).bfloat16()
    runs = []
    for table, scan in ((1023, B.VSA_STEP_SCAN_AHEAD), (1024, B.VSA_STEP_SCAN_AHEAD_MMA)):
        shape = B.make_shape(batch, 2, 1, table, 1024)
        assert B.vsa_step_scan(shape, P, 64) == scan
        bt = torch.arange(table, dtype=torch.int32, device=dev).expand(batch, -1).contiguous()
        dec = SparsePagedDecoder(shape, P, 64, 11.0, -float("inf"), device=dev)
        runs.append((dec, bt, dec.build_summaries(k, bt, lens)))
    us = [float("inf")] * 2
    for _ in range(10):
        for i, (dec, bt, summ) in enumerate(runs):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                dec.step(q, summ, k, k, bt, lens)
            b.record()
            torch.cuda.synchronize()
            us[i] = min(us[i], a.elapsed_time(b) * 50.0)
    assert us[1] < 1.08 * us[0], us
