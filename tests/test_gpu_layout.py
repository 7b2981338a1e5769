"""Speed that hangs on where the parts of a unit's shared memory start: the rows of the cache pass through it in 16-byte pieces, and off
the 128-byte lines they take a quarter more of the whole step."""
import pytest
import torch

from paper_2602_13804_b200 import SparsePagedDecoder
from paper_2602_13804_b200 import binding as B

pytestmark = pytest.mark.gpu


def test_time_grows_with_the_pages_only():
    """160 units of D = 256 with 46 pages against 40 (six rounds of tiles and five).  Off the lines 46 took 1.33 times as long,
    on them 1.10."""
    batch, table, dev = 5, 222, "cuda:0"
    gen = torch.Generator(device=dev).manual_seed(5)
    shape = B.make_shape(batch, 32, 8, table, batch * table, head_dim=256)
    k = torch.randn((batch * table, 8, 16, 256), generator=gen, device=dev).bfloat16()
    v = torch.randn((batch * table, 8, 16, 256), generator=gen, device=dev).bfloat16()
    q = torch.randn((batch, 32, 256), generator=gen, device=dev).bfloat16()
    bt = torch.randperm(batch * table, generator=gen, device=dev).int().view(batch, table)
    lens = torch.full((batch,), 3546, dtype=torch.int32, device=dev)
    runs = [SparsePagedDecoder(shape, P, 73, 16.0, -float("inf"), device=dev) for P in (40, 46)]
    summ = runs[0].build_summaries(k, bt, lens)
    us = [float("inf")] * 2
    for _ in range(10):
        for i, dec in enumerate(runs):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                dec.step(q, summ, k, v, bt, lens)
            b.record()
            torch.cuda.synchronize()
            us[i] = min(us[i], a.elapsed_time(b) * 50.0)
    assert us[1] < 1.2 * us[0], us
