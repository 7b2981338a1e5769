"""The token append right behind the kernel that advances the lengths (and, for one sequence, enters a page into the block
table): what it read ahead of its wait may be out of date, what it writes must not be."""
import pytest
import torch

from paper_2602_13804_b200 import binding as B

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("page", [16, 32])
@pytest.mark.parametrize("graph", [False, True])
def test_append_behind_the_length_update(page, graph):
    batch, hkv, pages, tokens = 6, 3, 8, 2 * page + 5
    gen = torch.Generator(device=DEV).manual_seed(11)
    pool = batch * pages + 1

    def randn(*shape):
        return torch.randn(shape, generator=gen, device=DEV).to(torch.bfloat16)
    k, v = randn(pool, hkv, page, 128), randn(pool, hkv, page, 128)
    k_ref, v_ref = k.clone(), v.clone()
    table = torch.randperm(pool, generator=gen, device=DEV)[: batch * pages].to(torch.int32).view(batch, pages)
    late = table[1].clone()
    table[1] = -1                                                # entered by the kernel in front of the append
    table[5, 1] = -1                                             # a page that does not exist: its tokens are dropped
    start = torch.tensor([0, page - 1, 1, page, 3 * page - 2, 5], dtype=torch.int32, device=DEV)
    lens = start.clone()
    shape = B.make_shape(batch, hkv, hkv, pages, pool, page_size=page)
    summ = torch.zeros((pool, hkv, 128), dtype=torch.bfloat16, device=DEV)
    k_new, v_new = randn(tokens, batch, hkv, 128), randn(tokens, batch, hkv, 128)
    k_in, v_in = k_new[0].clone(), v_new[0].clone()
    where = torch.zeros(1, dtype=torch.int64, device=DEV)

    def step():
        torch.index_select(k_new, 0, where, out=k_in.unsqueeze(0))
        torch.index_select(v_new, 0, where, out=v_in.unsqueeze(0))
        where.add_(1)
        table[1].copy_(late)
        lens.add_(1)
        B.vsa_append_kv(shape, k_in, v_in, k, v, table, lens, summ, None)

    if graph:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            step()
    for _ in range(tokens):
        g.replay() if graph else step()
    torch.cuda.synchronize()
    for t in range(tokens):
        for b in range(batch):
            at = int(start[b]) + t
            p = int(table[b, at // page])
            if p >= 0:
                k_ref[p, :, at % page], v_ref[p, :, at % page] = k_new[t, b], v_new[t, b]
    assert torch.equal(k, k_ref) and torch.equal(v, v_ref)
    want = torch.zeros_like(summ)
    B.vsa_build_page_summaries(shape, k_ref, table, lens, (start // page).to(torch.int32), want)
    torch.cuda.synchronize()
    assert torch.equal(summ, want)
