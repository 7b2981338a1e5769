"""Performance cases of the sparse paged decode step and of the cache maintenance around it.

A case is one pass of a decoding program: `layers` attention layers, each with its own paged K/V pools, page
summaries and queries, all sharing one block table and one set of sequence lengths, as the layers of a model do.

kind "decode": one decode step per layer through `SparsePagedDecoder` (or the fp8 entry point of the binding).
    call    "eager"  one Python call per layer, as a program that is still being written makes them
            "graph"  the same calls captured once into a CUDA graph and replayed, as a serving engine does
            "host"   q arrives in, and the results leave to, page-locked host memory (`step_host`)
    append  the step is preceded by the append of the token that is being decoded
    cache   "bf16", or "fp8" (e4m3 bytes with one power-of-two scale per page and KV head)
    solver  "closed" (softmax weights), "entropic" or "frank_wolfe" with `iters` iterations
kind "prefill": the page summaries (and with `radii` the page radii) of prompts that have just been written.

Lengths are spread log-uniformly from T_min to T_max over the batch.  `planted` of the sequences hold relevant
keys (the "needles" of the repository's workloads), one in every stretch of the context; sequences without them
have no support gap and take the dense pass.
"""
import math

import torch

from paper_2602_13804_b200 import SparsePagedDecoder
from paper_2602_13804_b200 import binding as B

DEVICE = "cuda:0"


def _decode(**more):
    case = dict(kind="decode", call="graph", layers=1, batch=1, n_q_heads=32, n_kv_heads=8, head_dim=128, page_size=16,
                T_min=4096, T_max=4096, P=32, K_c=256, planted=1.0, append=False, cache="bf16", solver="closed", iters=0)
    case.update(more)
    return case


def _prefill(**more):
    case = dict(kind="prefill", layers=1, batch=1, n_kv_heads=8, head_dim=128, page_size=16, T_min=4096, T_max=4096,
                cache="bf16", radii=False)
    case.update(more)
    return case


def listed():
    return [
        # one layer called from Python, short context: the smallest call, launches and host work
        _decode(name="layer_b1_t4k_eager", call="eager", T_min=4096, T_max=4096, P=16, K_c=128),
        # one chat user on a 32-layer model: append and step of every layer; the last page is partly filled
        _decode(name="token_b1_t4k", layers=32, T_min=4001, T_max=4001, append=True),
        # one user with a long document
        _decode(name="token_b1_t128k", layers=8, T_min=131072, T_max=131072, append=True),
        # the ordinary serving batch (the benchmark's workload)
        _decode(name="token_b8_t32k", layers=8, batch=8, T_min=32768, T_max=32768),
        # the same batch where q comes from, and the results go to, host memory
        _decode(name="host_b8_t32k", call="host", layers=8, batch=8, T_min=32768, T_max=32768),
        # long contexts for many users: the page scan has the largest share
        _decode(name="token_b16_t128k", batch=16, T_min=131072, T_max=131072),
        # ragged serving batch of a 70B-class model, eight query heads to a KV head
        _decode(name="ragged_b64_gqa8", batch=64, n_q_heads=64, T_min=4096, T_max=131072, P=64, K_c=512, append=True),
        # three sequences of four have no support gap: the dense pass
        _decode(name="fallback_b16_t64k", batch=16, T_min=65536, T_max=65536, planted=0.25),
        # e4m3 cache, a few sequences in the dense pass
        _decode(name="fp8_b16_t32k", layers=2, batch=16, T_min=16384, T_max=32768, planted=0.75, cache="fp8"),
        # small heads and 32-token pages, many short ragged sequences
        _decode(name="token_b32_t8k_d64", layers=4, batch=32, head_dim=64, page_size=32, T_min=1000, T_max=8191, P=16),
        # weights from four entropic iterations instead of the softmax
        _decode(name="solve_b8_t32k", layers=4, batch=8, T_min=32768, T_max=32768, solver="entropic", iters=4),
        # summaries of a batch of prompts
        _prefill(name="prefill_b8_t32k", layers=2, batch=8, T_min=8192, T_max=32768),
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        page_size = rng.choice((16, 16, 32))
        T_max = _log_between(rng, 1000, 131072)
        T_min = T_max if rng.random() < 0.4 else max(500, _log_between(rng, T_max / 16, T_max))
        batch = _log_between(rng, 1, 64)
        layers = _log_between(rng, 1, 32)
        if rng.random() < 0.12:
            case = _prefill(layers=layers, batch=batch, page_size=page_size, T_min=T_min, T_max=T_max,
                            n_kv_heads=rng.choice((1, 2, 8)), cache=rng.choice(("bf16", "bf16", "fp8")))
            if case["cache"] == "bf16":
                case["head_dim"] = rng.choice((64, 128, 128, 256))
                case["radii"] = case["head_dim"] == 128 and rng.random() < 0.5
        else:
            n_kv_heads, group = rng.choice(((8, 4), (8, 4), (8, 8), (32, 1), (16, 2), (2, 8), (1, 16)))
            P = _log_between(rng, 8, 2048 // page_size // 2)
            case = _decode(layers=layers, batch=batch, n_q_heads=n_kv_heads * group, n_kv_heads=n_kv_heads,
                           page_size=page_size, T_min=T_min, T_max=T_max, P=P,
                           K_c=min(P * page_size // 2, _log_between(rng, 64, 512)),
                           call=rng.choice(("eager", "graph", "graph", "graph", "host")),
                           planted=rng.choice((1.0, 1.0, 1.0, 0.75, 0.25)))
            option = rng.choice(("plain", "plain", "append", "append", "fp8", "head_dim", "solver"))
            if option == "append":
                case["append"] = True
            elif option == "fp8":
                case["cache"] = "fp8"
                case["call"] = rng.choice(("eager", "graph"))
            elif option == "head_dim":
                case["head_dim"] = rng.choice((64, 256))
            elif option == "solver":
                case["solver"] = rng.choice(("entropic", "frank_wolfe"))
                case["iters"] = rng.choice((2, 4, 6))
                case["K_c"] = min(case["K_c"], 256)
                case["call"] = rng.choice(("eager", "graph"))
        if _cost(case) <= most and _pool_bytes(case) <= 12e9:
            return case


# ---- sizes ---------------------------------------------------------------------------------------------

def _lengths(case):
    lo, hi, n = case["T_min"], case["T_max"], case["batch"]
    if n == 1:
        return [hi]
    return [int(round(lo * (hi / lo) ** (i / (n - 1)))) for i in range(n)]


def _pages(case):
    return [-(-t // case["page_size"]) for t in _lengths(case)]


def _pool_pages(case):
    used = sum(_pages(case))
    return used + used // 8 + 1


def _pool_bytes(case):
    element = 1 if case["cache"] == "fp8" else 2
    return case["layers"] * _pool_pages(case) * case["n_kv_heads"] * case["page_size"] * case["head_dim"] * 2 * element


def _planted(case):
    return [i < round(case.get("planted", 1.0) * case["batch"]) for i in range(case["batch"])]


def _decode_work(case):
    d, H, Hkv, page, P, K_c = (case[k] for k in ("head_dim", "n_q_heads", "n_kv_heads", "page_size", "P", "K_c"))
    element = 1 if case["cache"] == "fp8" else 2
    by = fl = 0.0
    for T, n, planted in zip(_lengths(case), _pages(case), _planted(case)):
        P_b = min(P, n)
        tokens = min(P_b * page, T)
        kept = min(K_c, tokens)
        by += n * (Hkv * d * 2 + 4)                              # every page summary, once, and its table entry
        by += Hkv * (tokens + kept) * d * element                # the routed pages' keys and the candidates' values
        by += H * (d * 2 + d * 4 + 32 + P * 4)                   # q; out, diag and routed pages
        fl += 2.0 * H * d * (n + tokens + kept)
        if case["solver"] != "closed":
            fl += 2.0 * H * d * kept * 2 * (case["iters"] + 1)
            by += H * 16
        if not planted and kept < T:                             # dense pass of the sequence's heads
            by += Hkv * (T - tokens) * d * element + Hkv * (T - kept) * d * element
            fl += 4.0 * H * T * d
        if case["append"]:
            by += Hkv * d * 2 * (2 + 2 + ((T - 1) % page) + 1)   # two rows in and out, the page's keys, its summary
            fl += Hkv * d * page
    return {"bytes": case["layers"] * by, "flops": case["layers"] * fl}


def work(case):
    """Bytes and operations of one pass: every input that the step has to look at once, every output once.
    The heads of a group are taken to route to the same pages, which is the least that they can read."""
    if case["kind"] == "decode":
        return _decode_work(case)
    element = 1 if case["cache"] == "fp8" else 2
    row = case["n_kv_heads"] * case["head_dim"]
    tokens, pages = sum(_lengths(case)), sum(_pages(case))
    by = row * (tokens * element + pages * 2) + 4 * pages
    fl = row * tokens
    if case["radii"]:
        by += 4 * pages * case["n_kv_heads"]
        fl += 3 * row * tokens
    return {"bytes": float(case["layers"] * by), "flops": float(case["layers"] * fl)}


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def tolerance(case):
    if case["kind"] == "prefill":
        return "exact"                              # fp32 sums in one stated order, rounded once
    # Routed pages, candidates, gaps and flags are the same numbers; `out` and `lse` are fp32 sums in any order, the
    # leakage bound an fp32 exponential of an argument up to about 100.  A unit of the dense pass has bf16
    # probabilities: many units where sequences lack planted keys, otherwise single ones at most.
    if not all(_planted(case)) or case["n_q_heads"] > 4 * case["n_kv_heads"] or case["head_dim"] == 64:
        return {"rel": 5e-3, "max": 0.05}
    return {"rel": 1e-3, "max": 0.05}


# ---- inputs --------------------------------------------------------------------------------------------

def _quantise(x):
    """e4m3 bytes and fp32 scales (the smallest power of two that fits a block) of x [pages, heads, page, d]."""
    amax = x.abs().amax(dim=(2, 3)).float().clamp(min=1e-30)
    scale = torch.exp2(torch.ceil(torch.log2(amax / 448.0)))
    scale = torch.where(amax / scale > 448.0, scale * 2, scale)
    return (x.float() / scale[:, :, None, None]).to(torch.float8_e4m3fn).view(torch.uint8), scale


def _pool(case, gen, needles=None):
    """One layer's K or V pool, filled with N(0, 1) rows; `needles`: (page, head, row, values) that overwrite it."""
    shape = (_pool_pages(case), case["n_kv_heads"], case["page_size"], case["head_dim"])
    x = torch.randn(shape, generator=gen, device=DEVICE, dtype=torch.bfloat16)
    if needles is not None:
        page, head, row, values = needles
        x[page, head, row] = values
    if case["cache"] == "bf16":
        return x, None
    bytes_, scales = torch.empty(shape, dtype=torch.uint8, device=DEVICE), []
    for at in range(0, shape[0], 8192):
        bytes_[at:at + 8192], s = _quantise(x[at:at + 8192])
        scales.append(s)
    return bytes_, torch.cat(scales)


def _table(case, gen):
    """Lengths in a random order with the sequences that hold relevant keys, and a random block table."""
    pages = _pages(case)
    order = torch.randperm(case["batch"], generator=gen, device=DEVICE).tolist()
    lens = [_lengths(case)[i] for i in order]
    planted = [_planted(case)[i] for i in order]
    free = torch.randperm(_pool_pages(case), generator=gen, device=DEVICE).to(torch.int32)
    table = torch.full((case["batch"], max(pages)), -1, dtype=torch.int32, device=DEVICE)
    at = 0
    for b, i in enumerate(order):
        table[b, :pages[i]] = free[at:at + pages[i]]
        at += pages[i]
    return lens, planted, table


def _needle_places(case, lens, planted, table, gen):
    """Where the relevant keys of one layer are: one in every P-th part of a planted sequence, per KV head."""
    n, Hkv, page = case["P"], case["n_kv_heads"], case["page_size"]
    seqs = [b for b in range(case["batch"]) if planted[b]]
    if not seqs:
        return None
    b = torch.tensor(seqs, device=DEVICE)[:, None, None].expand(-1, Hkv, n)
    g = torch.arange(Hkv, device=DEVICE)[None, :, None].expand(len(seqs), -1, n)
    T = torch.tensor([lens[s] for s in seqs], device=DEVICE, dtype=torch.float64)[:, None, None]
    part = torch.arange(n, device=DEVICE, dtype=torch.float64)
    u = torch.rand((len(seqs), Hkv, n), generator=gen, device=DEVICE, dtype=torch.float64)
    pos = ((part + u) * T / n).long().minimum(T.long() - 1)
    b, g, pos = b.reshape(-1), g.reshape(-1), pos.reshape(-1)
    return b, g, pos, table[b, pos // page].long(), pos % page


def _relevant_rows(q, case, b, g, gen):
    """Key rows that the query heads of KV head g of sequence b look for."""
    Hkv, G = case["n_kv_heads"], case["n_q_heads"] // case["n_kv_heads"]
    q_hat = q.float().view(case["batch"], Hkv, G, -1).sum(2)[b, g]
    noise = torch.randn(q_hat.shape, generator=gen, device=DEVICE)
    return (4.0 * q_hat + 0.1 * noise).to(torch.bfloat16)


def _outputs(case, state):
    """Views of everything the steps write, named; the record buffers split into their fields."""
    if case["kind"] == "prefill":
        return {k: state[k] for k in ("summaries", "radii") if k in state}
    diag = state["diag"]
    f = diag.view(torch.float32)
    out = {"out": state["out"], "delta": f[..., 0], "delta12": f[..., 1], "s_max": f[..., 2], "lse": f[..., 3],
           "leak_bound": f[..., 4], "n_candidates": diag[..., 5], "fallback": diag[..., 6], "status": diag[..., 7]}
    for k in ("routed_pages", "fallback_count", "solve"):
        if k in state:
            out[k] = state[k]
    if case["append"]:
        out["summaries"] = state["summaries"]
    return out


def prepare(case, seed):
    gen = torch.Generator(device=DEVICE).manual_seed(int(seed))
    L, batch, Hkv, d = case["layers"], case["batch"], case["n_kv_heads"], case["head_dim"]
    H = case.get("n_q_heads", Hkv)
    lens, planted, table = _table(case, gen)
    pool = _pool_pages(case)
    state = {"case": case, "table": table, "lens": torch.tensor(lens, dtype=torch.int32, device=DEVICE),
             "summaries": torch.zeros((L, pool, Hkv, d), dtype=torch.bfloat16, device=DEVICE), "steps": []}
    shape = B.make_shape(batch, H, Hkv, table.shape[1], pool, head_dim=d, page_size=case["page_size"])
    state["shape"] = shape

    if case["kind"] == "prefill":
        if case["radii"]:
            state["radii"] = torch.zeros((L, pool, Hkv), dtype=torch.float32, device=DEVICE)
        state["k"] = [_pool(case, gen) for _ in range(L)]
        state["outputs"] = _outputs(case, state)
        return state

    _prepare_decode(case, state, shape, lens, planted, gen)
    if case["call"] == "graph":
        _layers(state)                              # one pass ahead of the capture
        torch.cuda.synchronize()
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            _layers(state)
    return state


def _prepare_decode(case, state, shape, lens, planted, gen):
    L, batch, H, Hkv, d, P = (case[k] for k in ("layers", "batch", "n_q_heads", "n_kv_heads", "head_dim", "P"))
    host = case["call"] == "host"
    eps = math.sqrt(d)
    where = dict(device="cpu", pin_memory=True) if host else dict(device=DEVICE)
    # the layers' results side by side
    state["out"] = torch.zeros((L, batch, H, d), dtype=torch.float32, **where)
    state["diag"] = torch.zeros((L, batch * H, B.DIAG_BYTES // 4), dtype=torch.int32, **where)
    state["routed_pages"] = torch.zeros((L, batch, H, P), dtype=torch.int32, device=DEVICE)
    state["fallback_count"] = torch.zeros((L, 1), dtype=torch.int32, device=DEVICE)
    if case["solver"] != "closed":
        state["solve"] = torch.zeros((L, batch * H, 4), dtype=torch.float32, device=DEVICE)
    for i in range(L):
        q = torch.randn((batch, H, d), generator=gen, device=DEVICE).to(torch.bfloat16)
        places = _needle_places(case, lens, planted, state["table"], gen)
        needles = None
        if places is not None:
            b, g, _, page, row = places
            needles = (page, g, row, _relevant_rows(q, case, b, g, gen))
        k, k_scale = _pool(case, gen, needles)
        v, v_scale = _pool(case, gen)
        dec = SparsePagedDecoder(shape, P, case["K_c"], eps, 8.0 * eps, device=DEVICE)
        dec.routed_pages, dec.fallback_count = state["routed_pages"][i], state["fallback_count"][i]
        if host:
            dec.q_dev = torch.empty_like(q)
            dec.out_host, dec.diag_host = state["out"][i], state["diag"][i]
            q = q.cpu().pin_memory()
        else:
            dec.out, dec.diag = state["out"][i], state["diag"][i]
        if "solve" in state:
            dec.solve = state["solve"][i]
        if i:
            dec.ws = state["steps"][0]["dec"].ws    # one scratch buffer serves all layers
        s = {"dec": dec, "q": q, "k": k, "v": v, "k_scale": k_scale, "v_scale": v_scale, "summ": state["summaries"][i]}
        if case["append"]:                          # the new token attends to itself
            every = torch.arange(batch, device=DEVICE).repeat_interleave(Hkv)
            heads = torch.arange(Hkv, device=DEVICE).repeat(batch)
            q_dev = q.to(DEVICE)
            s["k_new"] = _relevant_rows(q_dev, case, every, heads, gen).view(batch, Hkv, d)
            noise = torch.randn((batch, Hkv, d), generator=gen, device=DEVICE).to(torch.bfloat16)
            without = torch.tensor([not p for p in planted], device=DEVICE)[:, None, None]
            s["k_new"] = torch.where(without, noise, s["k_new"])
            s["v_new"] = torch.randn((batch, Hkv, d), generator=gen, device=DEVICE).to(torch.bfloat16)
        if case["cache"] == "fp8":
            B.vsa_build_page_summaries_fp8(shape, k, k_scale, state["table"], state["lens"], None, s["summ"])
        else:
            dec.build_summaries(k, state["table"], state["lens"], None, s["summ"])
        state["steps"].append(s)
    state["outputs"] = _outputs(case, state)


# ---- one pass ------------------------------------------------------------------------------------------

def _layers(state):
    case, table, lens = state["case"], state["table"], state["lens"]
    for s in state["steps"]:
        dec = s["dec"]
        if case["append"]:
            dec.append(s["k_new"], s["v_new"], s["k"], s["v"], table, lens, s["summ"])
        if case["call"] == "host":
            dec.step_host(s["q"], s["summ"], s["k"], s["v"], table, lens)
        elif case["cache"] == "fp8":
            B.vsa_decode_step_fp8(dec.shape, s["q"], s["summ"], s["k"], s["v"], s["k_scale"], s["v_scale"], table, lens,
                                  dec.P, dec.K_c, dec.epsilon, dec.gap_threshold, dec.out, dec.diag, dec.routed_pages,
                                  dec.fallback_list, dec.fallback_count, dec.ws)
        elif case["solver"] == "entropic":
            dec.step_entropic(s["q"], s["summ"], s["k"], s["v"], table, lens, case["iters"])
        elif case["solver"] == "frank_wolfe":
            dec.step_frank_wolfe(s["q"], s["summ"], s["k"], s["v"], table, lens, case["iters"])
        else:
            dec.step(s["q"], s["summ"], s["k"], s["v"], table, lens)


def run(state):
    case = state["case"]
    if case["kind"] == "decode":
        if case["call"] == "graph":
            state["graph"].replay()
        else:
            _layers(state)
        return state["outputs"]
    for i, (k, k_scale) in enumerate(state["k"]):
        summ = state["summaries"][i]
        if case["cache"] == "fp8":
            B.vsa_build_page_summaries_fp8(state["shape"], k, k_scale, state["table"], state["lens"], None, summ)
        else:
            B.vsa_build_page_summaries(state["shape"], k, state["table"], state["lens"], None, summ)
        if case["radii"]:
            B.vsa_build_page_radii(state["shape"], k, summ, state["table"], state["lens"], None, state["radii"][i])
    return state["outputs"]
