"""Routed lists that name a page more than once (the contract asks for distinct pages): the page's tokens count once per
mention, as in the oracle, and the step stays inside its buffers - also for the last, partly filled page, and when the
cut between candidates and rejected tokens falls between the copies of one token."""
import numpy as np
import pytest
import torch

import oracle
from gpu_runner import check_out
from paper_2602_13804_b200 import binding as B
from util import geometry, host_arrays
from workloads import WorkloadSpec, make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,hq,hkv,P,K_c,d", [
    (3, 8, 2, 32, 75, 128),       # 512 threads
    (3, 8, 2, 128, 1000, 128),
    (20, 8, 4, 48, 301, 128),     # 256 threads
    (40, 8, 2, 64, 40, 128),      # 128 threads
    (40, 8, 2, 64, 500, 64),
    (3, 8, 2, 32, 75, 256),
])
def test_repeated_pages(batch, hq, hkv, P, K_c, d):
    lens = tuple(37 + 53 * (i % 11) for i in range(batch))   # every last page is partly filled
    w = make_workload(WorkloadSpec(name="rep", config=9, batch=batch, n_q_heads=hq, n_kv_heads=hkv, P=P, K_c=K_c,
                                   seq_lens=lens, needles=0, head_dim=d), seed=77 + P)
    rng = np.random.default_rng(5)
    routed = np.empty((batch, hq, P), np.int32)
    for b in range(batch):
        nb = -(-lens[b] // 16)
        routed[b] = rng.integers(-1, nb, (hq, P))
        routed[b, 0] = nb - 1            # the last page only
        routed[b, 1, : P // 2] = nb - 1
    dev = "cuda:0"
    wd = w.to(dev)
    shape = B.shape_of(wd.q, wd.k_cache, wd.block_table)
    units = batch * hq
    out = torch.full((batch, hq, d), float("nan"), dtype=torch.float32, device=dev)
    diag, flist = B.alloc_diag(units, dev), torch.empty(units, dtype=torch.int32, device=dev)
    fcount = torch.zeros(1, dtype=torch.int32, device=dev)
    B.vsa_sparse_decode(shape, wd.q, wd.k_cache, wd.v_cache, wd.block_table, wd.seq_lens,
                        torch.from_numpy(routed).to(dev), P, K_c, w.epsilon, w.gap_threshold, out, diag, flist, fcount)
    torch.cuda.synchronize()
    q, K, V, bt, sl = host_arrays(w)
    want = oracle.sparse(geometry(w), q, K, V, bt, sl, routed, K_c, w.epsilon, w.gap_threshold)
    check_out(out.cpu().numpy(), want.out, "out")
    got = B.diag_to_dict(diag)
    for name in ("delta", "delta12", "s_max", "n_candidates", "fallback"):
        assert np.array_equal(got[name].numpy().reshape(batch, hq), getattr(want, name)), name
