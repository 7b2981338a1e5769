"""A stream that has a few of the device's SMs only (a green context), too few in one place for the clusters in which a step scans its
pages: the step takes the scan ahead there, with the results of the whole device."""
import pytest
import torch

from paper_2602_13804_b200 import binding as B
from test_gpu_page_mma import _workload

pytestmark = pytest.mark.gpu


@pytest.fixture
def few_sms():
    """A stream with eight SMs that share no GPC, or no more than the two of a TPC: no cluster of four blocks of one SM each."""
    drv = pytest.importorskip("cuda.bindings.driver")
    torch.zeros(1, device="cuda:0")

    def ok(result):
        if int(result[0]) != 0:
            pytest.skip(f"no green contexts here: {result[0]}")
        return result[1] if len(result) == 2 else result[1:]

    dev = ok(drv.cuDeviceGet(0))
    sms = ok(drv.cuDeviceGetDevResource(dev, drv.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM))
    loose = drv.CUdevSmResourceSplit_flags.CU_DEV_SM_RESOURCE_SPLIT_IGNORE_SM_COSCHEDULING
    parts, _, _ = ok(drv.cuDevSmResourceSplitByCount(1, sms, int(loose), 8))
    ctx = ok(drv.cuGreenCtxCreate(ok(drv.cuDevResourceGenerateDesc(parts, 1)), dev,
                                  drv.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM))
    stream = ok(drv.cuGreenCtxStreamCreate(ctx, drv.CUstream_flags.CU_STREAM_NON_BLOCKING, 0))
    yield int(stream), lambda: ok((*drv.cuStreamSynchronize(stream), None))
    drv.cuStreamDestroy(stream)
    drv.cuGreenCtxDestroy(ctx)


@pytest.mark.parametrize("batch,hq,hkv,table,kind,scan", [
    (1, 32, 8, 256, "closed", "INSIDE"),
    (4, 32, 8, 4096, "closed", "INSIDE_MMA"),
    (10, 16, 2, 600, "closed", "INSIDE_MMA"),
    (4, 32, 8, 2048, "entropic", "INSIDE_MMA"),
])
def test_step_on_few_sms(few_sms, batch, hq, hkv, table, kind, scan):
    stream, wait = few_sms
    w = _workload(batch, hq, hkv, 600)
    w.seq_lens.clamp_(max=16 * min(table, 600))
    w.block_table = torch.nn.functional.pad(w.block_table[:, :table], (0, max(0, table - 600)), value=-1).contiguous()
    wd = w.to("cuda:0")
    shape, units, P, K_c = B.shape_of(wd.q, wd.k_cache, wd.block_table), batch * hq, 24, 100
    solve = kind == "entropic"
    assert B.vsa_step_scan(shape, P, K_c, B.VSA_STEP_SOLVE if solve else B.VSA_STEP_CLOSED) == getattr(B, "VSA_STEP_SCAN_" + scan)
    summ = torch.zeros((shape.num_pool_pages, hkv, 128), dtype=torch.bfloat16, device="cuda:0")
    B.vsa_build_page_summaries(shape, wd.k_cache, wd.block_table, wd.seq_lens, None, summ)

    def run(on):
        out, diag, sol = torch.empty_like(wd.q, dtype=torch.float32), B.alloc_diag(units, "cuda:0"), B.alloc_solve(units, "cuda:0")
        routed = torch.empty((batch, hq, P), dtype=torch.int32, device="cuda:0")
        flist, fcount = torch.full((units,), -1, dtype=torch.int32, device="cuda:0"), torch.zeros(1, dtype=torch.int32, device="cuda:0")
        ws = B.alloc_workspace(shape, P, K_c, B.VSA_WS_STEP, "cuda:0")
        torch.cuda.synchronize()
        args = (shape, wd.q, summ, wd.k_cache, wd.v_cache, wd.block_table, wd.seq_lens, P, K_c, w.epsilon, w.gap_threshold)
        rest = (routed, flist, fcount, ws, on)
        if solve:
            B.vsa_decode_step_entropic(*args, 3, out, diag, sol, *rest)
        else:
            B.vsa_decode_step(*args, out, diag, *rest)
        if on is not None:
            wait()
        torch.cuda.synchronize()
        return out, B.diag_to_dict(diag), routed, flist.sort().values

    whole, few = run(None), run(stream)
    assert torch.equal(whole[2], few[2]) and torch.equal(whole[3], few[3])
    for name, want in whole[1].items():
        if name not in ("lse", "leak_bound"):
            assert torch.equal(few[1][name], want), name
    # sums of up to 100 weights of at most 1 (and of values of a few units) in another order: 100 * 2^-24 * 5 at most
    assert float((few[0] - whole[0]).abs().max()) <= 1e-4
