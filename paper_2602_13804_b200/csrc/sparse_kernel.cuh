// Fused sparse pass of the routing variants (kernel template and its launch dispatch; included by the translation
// units that instantiate one of them each): the routing certificate (sparse_cert.cu), which needs every page score of
// the unit in registers, and the two-level front end (sparse_two_level.cu).  The closed-form step and the iterative
// solves are in sparse_step.cuh.
// One (sequence, query head) unit per thread block (paper Sec. 7 steps 2-4, Sec. 8 gap statistic, Cor. 1 leakage
// bound, Sec. 10.3 fallback flag):
//   top-P page selection -> score every valid token of the routed pages -> exact top-K_c -> softmax weights at
//   temperature epsilon -> weighted sum of the candidates' value rows -> diagnostics.
// The candidate list and the weights live in shared memory and registers only.
#pragma once

#include <limits.h>
#include <math.h>

#include "vsa_device.cuh"
#include "vsa_launch.h"
#include "vsa_select.cuh"

namespace vsa {

namespace {


constexpr int kMaxSparseWarps = 16;

// token-phase shared memory, in 4-byte words, after the two tile arrays (PT = routed tiles of 16 tokens)
__host__ __device__ constexpr int token_phase_words(int PT, int K_c)
{
    return PT * 16 /*keys*/ + (PT * 16 + 3) / 4 /*take*/ + 2 * K_c + 2 /*voff*/ + K_c /*wgt*/ +
           256 + 16 + 72 + kTopkList + kMaxSparseWarps * kHeadDim + kMaxSparseWarps + 4;
}

// first word of the block-table copy: after the two tile arrays and the larger of the two phases
__host__ __device__ inline int bt_stage_offset_words(int max_pages, int P, int PT, int K_c)
{
    int words = token_phase_words(PT, K_c);
    if (select_pages_words(max_pages, P) > words) words = select_pages_words(max_pages, P);
    return 2 * PT + words;
}

// Two-level front end (PAGE_KPT == -2): [selection over the super-pages | exact keys of the pages inside the
// kept super-pages, 16 per super-page | selection over those], all dead before the token phase
__host__ __device__ inline int two_level_words(int max_pages, int P, int P_super)
{
    const int max_supers = (max_pages + 15) / 16;
    return select_pages_words(max_supers, P_super) + 16 * P_super + select_pages_words(16 * P_super, P);
}
__host__ __device__ inline int two_level_smem_words(int max_pages, int P, int PT, int K_c, int P_super)
{
    const int a = token_phase_words(PT, K_c), b = two_level_words(max_pages, P, P_super);
    return 2 * PT + (a > b ? a : b);
}

struct TokenSmem {
    uint32_t* keys;   // [PT * 16] token score keys, array index = 16 * slot + token (position order)
    uint8_t* take;    // [PT * 16] scratch of the selection's slow path
    long long* voff;  // [K_c] element offset of each candidate's value row, candidates in position order
    float* wgt;       // [K_c] unnormalised softmax weight of each candidate
    TopkScratch ts;
    float* red;       // [warps][128]
    float* zred;      // [warps]
};

__device__ __forceinline__ TokenSmem carve_tokens(uint32_t* base, int PT, int K_c)
{
    TokenSmem s;
    const int N = PT * 16;
    s.keys = base;
    s.take = (uint8_t*)(s.keys + N);
    uint32_t* after_take = s.keys + N + (N + 3) / 4;
    after_take += ((uintptr_t)after_take & 4u) ? 1 : 0;   // 8-byte alignment of the offsets
    s.voff = (long long*)after_take;
    s.wgt = (float*)(s.voff + K_c);
    s.ts.hist = (uint32_t*)(s.wgt + K_c);
    s.ts.misc = s.ts.hist + 256;
    s.ts.wred = s.ts.misc + 16;
    s.ts.list = (int32_t*)(s.ts.wred + 72);
    s.red = (float*)(s.ts.list + kTopkList);
    s.zred = s.red + kMaxSparseWarps * kHeadDim;
    return s;
}

__device__ __forceinline__ void write_failed_unit(float* out, vsa_diag_t* diag, long long unit, int status)
{
    for (int e = threadIdx.x; e < kHeadDim; e += blockDim.x) out[unit * kHeadDim + e] = 0.0f;
    if (threadIdx.x == 0) {
        vsa_diag_t d;
        d.delta = d.delta12 = d.s_max = d.lse = d.leak_bound = 0.0f;
        d.n_candidates = 0;
        d.fallback = 0;
        d.status = status;
        diag[unit] = d;
    }
}

// THREADS: 256 (two blocks per SM; the throughput shape), 512 (one block per SM; used when there
//   are no more units than SMs, so that one unit gets twice the loads in flight and half the passes)
//   or 128 (four blocks per SM; used when there are more units than two blocks per SM hold: more
//   units in flight, fewer waves).
// PAGE_KPT == -2: fused with two-level routing; page_scores holds the unit's scores of the super-pages'
//   representatives [unit][ceil(max_pages / 16)]; the P_super best super-pages are kept, the pages inside
//   them scored exactly from tl_summaries, and the top-P of those routed.
// PAGE_KPT  >  0: each thread keeps PAGE_KPT page scores in registers.
//   In both forms the unit's top-P pages are selected here from page_scores[unit][0..n_b) and written to
//   routed_pages (best first, -1 padded).
// TOK_KPT: token scores per thread, P * 16 <= TOK_KPT * THREADS.
// CERT (fused register variants only): the certified gap of the unit - an upper bound on every score
//   of the pages that were not routed, from the pages' radii (rad_logical, written by the scan) -
//   is computed, reported in cert[] and used for the fallback decision in place of the proxy gap.
template <int THREADS, int PAGE_KPT, int TOK_KPT, bool CERT>
__global__ void __launch_bounds__(THREADS, 512 / THREADS)
sparse_decode_kernel(Geometry geo, const uint16_t* __restrict__ q, const uint16_t* __restrict__ k_cache,
                     const uint16_t* __restrict__ v_cache, const int32_t* __restrict__ block_table,
                     const int32_t* __restrict__ seq_lens, int32_t* __restrict__ routed_pages,
                     const float* __restrict__ page_scores, int P, int K_c, float epsilon, float gap_threshold,
                     float* __restrict__ out, vsa_diag_t* __restrict__ diag, int32_t* __restrict__ fallback_list,
                     int32_t* __restrict__ fallback_count,
                     const float* __restrict__ rad_logical, vsa_cert_t* __restrict__ cert,
                     const int32_t* __restrict__ unit_list, const int32_t* __restrict__ unit_count,
                     int routed_stride,
                     const uint16_t* __restrict__ tl_summaries, int P_super)
{
    constexpr int WARPS = THREADS / 32, GROUPS = 2 * WARPS;
    static_assert(PAGE_KPT > 0 || (PAGE_KPT == -2 && !CERT), "two-level front end: no certificate");
    static_assert(!CERT || PAGE_KPT > 0, "the certificate needs every page score of the unit in registers");
    static_assert(TOK_KPT * WARPS <= 64 && 4 * WARPS <= 72, "wred capacity");
    extern __shared__ uint32_t smem_raw[];
    // The token phases work on tiles of 16 rows: a routed page is 1 << tile_shift of them (one at 16 tokens
    // per page, two at 32).  Tile v of the sequence holds tokens 16 v .. 16 v + 15.
    const int tsh = geo.tile_shift, PT = P << tsh;
    int32_t* page_l = (int32_t*)smem_raw;   // [PT] tiles of the routed pages, ascending, invalid entries last
    int32_t* page_phys = page_l + PT;       // [PT] pool page of each tile
    uint32_t* region = smem_raw + 2 * PT;   // page-selection scratch first, token-phase arrays afterwards
    const int N = PT * 16;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = lane & 15, gi = lane >> 4;
    // unit_list != nullptr: block i handles unit_list[i] for i < *unit_count (a retry pass over the units
    // an earlier pass of the same step listed); the list is that pass's product, so it is read after
    // the wait
    long long unit = blockIdx.x;
    if (unit_list) {
        pdl_wait();
        if ((int)blockIdx.x >= __ldcg(unit_count)) {
            pdl_launch_dependents();
            return;
        }
        unit = __ldcg(unit_list + blockIdx.x);
    }
    const int b = (int)(unit / geo.n_q_heads), h = (int)(unit % geo.n_q_heads), g = h / geo.group;
    // Loads that depend on nothing computed in this step go out before the wait on the preceding
    // kernel: the sequence length, the query row (the routing kernel that precedes this one in a step
    // has read it already) and a copy of the block-table row for the page lookups that follow the
    // selection.  The page scores, which that kernel writes, are fetched right after the wait (the
    // sequence length, asked for before it, has arrived by then).
    const int32_t* bt = block_table + (long long)b * geo.max_pages;
    const int T = ld_ca_s32(seq_lens + b);
    const uint4 qraw = ld_nc_16B(q + unit * kHeadDim + c * 8);
    int32_t* bt_s = (int32_t*)(smem_raw + bt_stage_offset_words(geo.max_pages, P, PT, K_c));
    if constexpr (PAGE_KPT > 0) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(bt_s);
        for (int i = tid; i < geo.max_pages; i += THREADS) cp_async_4(dst + 4u * (uint32_t)i, bt + i);
        cp_async_commit_group();
    }
    pdl_wait();
    pdl_launch_dependents();
    // Only the scores of the sequence's own pages are fetched: the rest of the scratch row was not
    // written in this step (in a ragged batch it is most of the row, and it would come from DRAM).
    const int nb_fetch = geo.length_ok(T) ? geo.pages_of(T) : 0;
    float praw[PAGE_KPT > 0 ? PAGE_KPT : 1];
    if constexpr (PAGE_KPT > 0) {
#pragma unroll
        for (int j = 0; j < PAGE_KPT; ++j) {
            const int i = tid + j * THREADS;
            praw[j] = i < nb_fetch ? ld_cg_f32(page_scores + unit * geo.max_pages + i) : 0.0f;
        }
    }
    float prad[CERT ? PAGE_KPT : 1];
    if constexpr (CERT) {
#pragma unroll
        for (int j = 0; j < PAGE_KPT; ++j) {
            const int i = tid + j * THREADS;
            prad[j] = i < nb_fetch
                          ? ld_cg_f32(rad_logical + ((long long)b * geo.n_kv_heads + g) * geo.max_pages + i)
                          : 0.0f;
        }
    }
    if (!geo.length_ok(T)) {
        cp_async_wait_all();
        write_failed_unit(out, diag, unit, VSA_UNIT_BAD_LENGTH);
        if (CERT && tid == 0) cert[unit] = vsa_cert_t{0.0f, 0.0f, 0.0f, 0};
        for (int t = tid; t < routed_stride; t += THREADS) routed_pages[unit * routed_stride + t] = -1;
        return;
    }
    const int nb = geo.pages_of(T);

    // ---- routed pages -> page_l[] sorted by logical page, so that array order = position order ----
    int np;
    int bad = 0;
    {
        const PageSelectSmem ps =
            PAGE_KPT == -2 ? carve_page_select(region + select_pages_words((geo.max_pages + 15) >> 4, P_super) + 16 * P_super,
                                               16 * P_super, P)
                           : carve_page_select(region, geo.max_pages, P);
        if constexpr (PAGE_KPT > 0) {
            uint32_t pkey[PAGE_KPT];
#pragma unroll
            for (int j = 0; j < PAGE_KPT; ++j)
                pkey[j] = tid + j * THREADS < nb ? float_to_key(praw[j]) : 0u;
            cp_async_wait_all();   // this thread's part of the block-table copy; the selection's barriers publish it
            np = select_top_pages_keys<PAGE_KPT>(pkey, nb, P, ps);
            if constexpr (CERT) {
                // |q| (rounded up a little), every lane of a half-warp computing the same value
                float qe[8];
                unpack8(qraw, qe);
                float q2 = chunk_partial(qe, qe);
#pragma unroll
                for (int off = 8; off; off >>= 1) q2 = q2 + __shfl_xor_sync(kFullMask, q2, off);
                const float qn = __fmul_rn(__fsqrt_rn(q2), 1.00000095367431640625f);
                // a page is un-routed iff it is ordered after the last winner (score descending, index
                // ascending); its tokens score at most  c + |q| * radius
                const uint32_t k_last = ps.win_key[np - 1];
                const int i_last = ps.win_idx[np - 1];
                uint32_t ub_key = 0u;
#pragma unroll
                for (int j = 0; j < PAGE_KPT; ++j) {
                    const int i = tid + j * THREADS;
                    const bool unrouted = pkey[j] != 0u && ((pkey[j] < k_last) | ((pkey[j] == k_last) & (i > i_last)));
                    if (unrouted)
                        ub_key = max(ub_key, float_to_key(__fadd_rn(key_to_float(pkey[j]), __fmul_rn(qn, prad[j]))));
                }
                ub_key = __reduce_max_sync(kFullMask, ub_key);
                if (lane == 0) ps.ts.wred[warp] = ub_key;   // published by the barrier below, read right after it
            }
        }
        // position -> logical page of a winner (two-level: position 16 j + c is page c of the j-th kept
        // super-page in ascending order)
        const int32_t* asc_super = nullptr;
        if constexpr (PAGE_KPT == -2) {
            const int max_supers = (geo.max_pages + 15) >> 4, ns = (nb + 15) >> 4;
            const PageSelectSmem ps1 = carve_page_select(region, max_supers, P_super);
            uint32_t* exact = region + select_pages_words(max_supers, P_super);
            uint32_t skey[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int i = tid + j * THREADS;
                skey[j] = i < ns ? float_to_key(ld_cg_f32(page_scores + unit * max_supers + i)) : 0u;
            }
            if (tid == 0) ps1.ts.misc[12] = 0u;   // pages that get a score (a word the selection does not use)
            const int Ks = select_top_pages_keys<8>(skey, ns, P_super, ps1);   // ends with a barrier
            asc_super = ps1.asc_idx;
            float qe[8];
            unpack8(qraw, qe);
            // one kept super-page = 16 summary rows = one 16-value reduction per half-warp; lane c ends with
            // the exact score of page 16 s + c
            for (int j0 = warp * 2; j0 < Ks; j0 += GROUPS) {
                const int j = j0 + gi;
                const bool have = j < Ks;
                const int l = have ? asc_super[j] * 16 + c : nb;
                long long phys = -1;
                if (l < nb) {
                    phys = bt[l];
                    if (phys < 0 || phys >= geo.pool_pages) phys = -1;
                }
                uint4 srows[16];
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    const long long pr = __shfl_sync(kFullMask, phys, (lane & 16) | r);
                    srows[r] = pr >= 0 ? ld_nc_16B(tl_summaries + (pr * geo.n_kv_heads + g) * kHeadDim + c * 8)
                                       : make_uint4(0u, 0u, 0u, 0u);
                }
                float vals[16];
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    float kf[8];
                    unpack8(srows[r], kf);
                    vals[r] = chunk_partial(qe, kf);
                }
                const float sc = reduce_scatter16(vals, c);
                const bool scored = have && phys >= 0;
                if (have) exact[j * 16 + c] = scored ? float_to_key(sc) : 0u;
                const int n_ok = __popc(__ballot_sync(kFullMask, scored));
                if (lane == 0 && n_ok) atomicAdd(&ps1.ts.misc[12], (uint32_t)n_ok);
            }
            __syncthreads();
            const int n2 = Ks * 16, P2 = min(P, (int)ps1.ts.misc[12]);
            uint32_t pkey2[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int i = tid + j * THREADS;
                pkey2[j] = i < n2 ? exact[i] : 0u;
            }
            np = P2 > 0 ? select_top_pages_keys<8>(pkey2, n2, P2, ps) : 0;
        }
        auto page_of = [&](int pos) { return PAGE_KPT == -2 ? asc_super[pos >> 4] * 16 + (pos & 15) : pos; };
        for (int t = P + tid; t < routed_stride; t += THREADS) routed_pages[unit * routed_stride + t] = -1;
        for (int t = tid; t < P; t += THREADS) {
            routed_pages[unit * routed_stride + t] = t < np ? page_of(ps.win_idx[t]) : -1;
            int l = INT_MAX, phys = -1;
            if (t < np) {
                l = page_of(ps.asc_idx[t]);
                phys = PAGE_KPT > 0 ? bt_s[l] : bt[l];
                if (phys < 0 || phys >= geo.pool_pages) {
                    phys = -1;
                    bad = 1;
                }
            }
            for (int hf = 0; hf < (1 << tsh); ++hf) {
                page_l[(t << tsh) + hf] = l == INT_MAX ? INT_MAX : (l << tsh) + hf;
                page_phys[(t << tsh) + hf] = phys;
            }
        }
    }
    const int any_bad = __syncthreads_or(bad);
    uint32_t ub_unrouted_key = 0u;   // CERT: key of the best upper bound over the un-routed pages, 0 = none
    if constexpr (CERT) {
        const PageSelectSmem ps = carve_page_select(region, geo.max_pages, P);
#pragma unroll
        for (int w = 0; w < WARPS; ++w) ub_unrouted_key = max(ub_unrouted_key, ps.ts.wred[w]);
        __syncthreads();   // the selection scratch is rewritten by the token phase
    }
    if (any_bad) {
        write_failed_unit(out, diag, unit, VSA_UNIT_BAD_PAGE);
        if (CERT && tid == 0) cert[unit] = vsa_cert_t{0.0f, 0.0f, 0.0f, 0};
        return;
    }
    const TokenSmem sm = carve_tokens(region, PT, K_c);
    const int nt = np << tsh;   // tiles of the routed pages
#pragma unroll
    for (int j = 0; j < TOK_KPT; ++j)
        if (tid + j * THREADS < N) sm.keys[tid + j * THREADS] = 0u;
    __syncthreads();

    // ---- token routing: score all 16 tokens of a page per half-warp ----
    float qf[8];
    unpack8(qraw, qf);
    for (int pp = warp; pp * 2 < nt; pp += WARPS) {
        const int slot = pp * 2 + gi;
        const bool active = slot < nt;
        float vals[16];
        uint4 rows[16];
        if (active) {
            const uint16_t* src = k_cache + (long long)page_phys[slot] * geo.page_stride + (long long)g * geo.head_stride +
                                  c * 8 + (long long)((page_l[slot] & ((1 << tsh) - 1)) * 16) * geo.token_stride;
#pragma unroll
            for (int t = 0; t < 16; ++t) rows[t] = ld_nc_16B(src + (long long)t * geo.token_stride);
        } else {
#pragma unroll
            for (int t = 0; t < 16; ++t) rows[t] = make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            float kf[8];
            unpack8(rows[t], kf);
            vals[t] = chunk_partial(qf, kf);
        }
        const float s = reduce_scatter16(vals, c);   // lane c: score of token c of the page
        if (active && page_l[slot] * 16 + c < T) sm.keys[slot * 16 + c] = float_to_key(s);
    }
    __syncthreads();

    // ---- every thread takes its TOK_KPT token keys into registers ----
    uint32_t key[TOK_KPT];
    int present = 0;
    uint32_t a1 = 0u, a2 = 0u;   // best and second-best key (multiset order statistics)
    uint32_t amin = 0xffffffffu;  // smallest present key
#pragma unroll
    for (int j = 0; j < TOK_KPT; ++j) {
        const int i = tid + j * THREADS;
        key[j] = i < N ? sm.keys[i] : 0u;
        present += key[j] != 0u;
        if (key[j] != 0u) amin = min(amin, key[j]);
        if (key[j] > a1) {
            a2 = a1;
            a1 = key[j];
        } else if (key[j] > a2) {
            a2 = key[j];
        }
    }
    // number of valid scored tokens, the two best keys and the smallest key: per warp with the
    // single-instruction warp reductions, then across the warps through shared memory.  Each warp
    // also publishes its best key: the smallest of those (hi_r) and the largest of the warps' smallest
    // keys (lo_r) bracket the bulk of the scores and serve as the histogram range of the selection.
    {
        present = __reduce_add_sync(kFullMask, present);
        amin = __reduce_min_sync(kFullMask, amin);
        const uint32_t wmax = __reduce_max_sync(kFullMask, a1);
        const int holder = __ffs(__ballot_sync(kFullMask, a1 == wmax)) - 1;
        const uint32_t wsecond = __reduce_max_sync(kFullMask, lane == holder ? a2 : a1);
        a1 = wmax;
        a2 = wsecond;
    }
    if (lane == 0) {
        sm.ts.wred[4 * warp] = a1;
        sm.ts.wred[4 * warp + 1] = a2;
        sm.ts.wred[4 * warp + 2] = (uint32_t)present;
        sm.ts.wred[4 * warp + 3] = amin;
    }
    // the selection below starts from a cleared histogram and list counter
    for (int i = tid; i < 256; i += THREADS) sm.ts.hist[i] = 0u;
    if (tid == 0) sm.ts.misc[4] = 0u;
    __syncthreads();
    uint32_t key1 = 0u, key2 = 0u, kmin = 0xffffffffu, hi_r = 0xffffffffu, lo_r = 0u;
    int n_valid = 0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
        const uint32_t b1 = sm.ts.wred[4 * w], b2 = sm.ts.wred[4 * w + 1], bmin = sm.ts.wred[4 * w + 3];
        const uint32_t n1 = max(key1, b1), n2 = max(min(key1, b1), max(key2, b2));
        key1 = n1;
        key2 = n2;
        n_valid += (int)sm.ts.wred[4 * w + 2];
        kmin = min(kmin, bmin);
        if (b1 != 0u) hi_r = min(hi_r, b1);                 // warps without a valid token do not count
        if (bmin != 0xffffffffu) lo_r = max(lo_r, bmin);
    }
    const int ns = min(K_c, n_valid);

    // ---- exact top-(ns+1): its last element is the best rejected token, the rest are the candidates ----
    uint32_t out_key = 0u, mask = 0u;
    const bool has_rejected = n_valid > ns;
    if (has_rejected) {
        // token scores are finite, so the smallest and largest keys are the range of the finite scores
        // (when the bracket is empty or inverted the selection falls back to the full range itself)
        const TopkRegResult r = block_topk_reg<TOK_KPT, true>(key, N, ns + 1, sm.ts, sm.keys, sm.take,
                                                             key_to_float(lo_r), key_to_float(hi_r),
                                                             key_to_float(kmin), key_to_float(key1));
        out_key = r.kth_key;
        mask = r.mask;
#pragma unroll
        for (int j = 0; j < TOK_KPT; ++j)
            if (tid + j * THREADS == r.kth_idx) mask &= ~(1u << j);
    } else {
#pragma unroll
        for (int j = 0; j < TOK_KPT; ++j)
            if (key[j] != 0u) mask |= 1u << j;
        __syncthreads();   // wred is rewritten by the compaction
    }

    // ---- ordered compaction of the candidates (position order); the thread that holds a candidate's
    //      key writes the address of its value row and its softmax weight ----
    const float s1 = ns > 0 ? key_to_float(key1) : -INFINITY;
    const float scale = 1.4426950408889634f / epsilon;   // log2(e) / epsilon
    {
        int before[TOK_KPT];
#pragma unroll
        for (int j = 0; j < TOK_KPT; ++j) {
            const unsigned bal = __ballot_sync(kFullMask, (mask >> j) & 1u);
            before[j] = __popc(bal & ((1u << lane) - 1u));
            if (lane == 0) sm.ts.wred[j * WARPS + warp] = (uint32_t)__popc(bal);
        }
        __syncthreads();
        int base = 0;
#pragma unroll
        for (int j = 0; j < TOK_KPT; ++j) {
            // elements of row j (indices j * THREADS + tid) come after all of rows < j
            int mine = base;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) {
                const int cw = (int)sm.ts.wred[j * WARPS + w];
                if (w < warp) mine += cw;
                base += cw;
            }
            if ((mask >> j) & 1u) {
                const int i = tid + j * THREADS, pos = mine + before[j];
                sm.voff[pos] = (long long)page_phys[i >> 4] * geo.page_stride +
                               (long long)((page_l[i >> 4] & ((1 << tsh) - 1)) * 16 + (i & 15)) * geo.token_stride;
                sm.wgt[pos] = exp2f((key_to_float(key[j]) - s1) * scale);
            }
        }
    }
    __syncthreads();

    // ---- value gather ----
    float acc[8], z = 0.0f;
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
    const int gidx = warp * 2 + gi;
    constexpr int UNR = THREADS == 512 ? 8 : 16;   // 256 threads, K_c = 256: every half-warp's rows in one batch
    const uint16_t* vbase = v_cache + (long long)g * geo.head_stride + c * 8;
    for (int j0 = gidx; j0 < ns; j0 += GROUPS * UNR) {
        // all value rows of the batch at once; slots past the candidate count re-read the last candidate with weight 0
        uint4 rows[UNR];
        float w[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            const int j = j0 + u * GROUPS, jc = min(j, ns - 1);
            rows[u] = ld_nc_16B(vbase + sm.voff[jc]);
            w[u] = j < ns ? sm.wgt[jc] : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            float vf[8];
            unpack8(rows[u], vf);
#pragma unroll
            for (int e = 0; e < 8; e += 2) fma2(acc[e], acc[e + 1], w[u], w[u], vf[e], vf[e + 1]);
            z += w[u];
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] += __shfl_xor_sync(kFullMask, acc[e], 16);
    z += __shfl_xor_sync(kFullMask, z, 16);
    if (gi == 0) {
#pragma unroll
        for (int e = 0; e < 8; ++e) sm.red[warp * kHeadDim + c * 8 + e] = acc[e];
        if (c == 0) sm.zred[warp] = z;
    }
    __syncthreads();
    float Z = 0.0f;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) Z += sm.zred[w];
    for (int e = tid; e < kHeadDim; e += THREADS) {
        float a = 0.0f;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) a += sm.red[w * kHeadDim + e];
        out[unit * kHeadDim + e] = ns > 0 ? a / Z : 0.0f;
    }

    // ---- diagnostics and fallback flag ----
    if (tid == 0) {
        const float s2 = ns > 1 ? key_to_float(key2) : -INFINITY;
        const float delta = has_rejected ? s1 - key_to_float(out_key) : INFINITY;
        vsa_diag_t d;
        d.delta = delta;
        d.delta12 = ns > 0 ? s1 - s2 : INFINITY;
        d.s_max = s1;
        d.lse = ns > 0 ? s1 / epsilon + logf(Z) : -INFINITY;
        d.leak_bound = fminf(1.0f, (float)(T - ns) * expf(-delta / epsilon));
        d.n_candidates = ns;
        d.fallback = (delta < gap_threshold && ns < T) ? 1 : 0;
        if constexpr (CERT) {
            const float ub = ub_unrouted_key != 0u ? key_to_float(ub_unrouted_key) : -INFINITY;
            const float rej = has_rejected ? key_to_float(out_key) : -INFINITY;
            const float m = fmaxf(rej, ub);
            vsa_cert_t ce;
            ce.ub_unrouted = ub;
            ce.delta_cert = m == -INFINITY ? INFINITY : s1 - m;
            ce.certified = ce.delta_cert >= gap_threshold ? 1 : 0;
            ce.leak_bound_cert = fminf(1.0f, (float)(T - ns) * expf(-ce.delta_cert / epsilon));
            cert[unit] = ce;
            d.fallback = (!ce.certified && ns < T) ? 1 : 0;   // the certified gap decides
        }
        d.status = 0;
        diag[unit] = d;
        if (d.fallback) fallback_list[atomicAdd(fallback_count, 1)] = (int32_t)unit;
    }
}

}  // namespace

// everything one launch of the fused kernel needs
struct SparseArgs {
    Geometry g;
    size_t smem;
    const uint16_t *q, *k, *v;
    const int32_t *block_table, *seq_lens;
    int32_t* routed_pages;
    const float* page_scores;
    int P, K_c;
    float epsilon, gap_threshold;
    float* out;
    vsa_diag_t* diag;
    int32_t *fallback_list, *fallback_count;
    const float* rad_logical;
    vsa_cert_t* cert;     // non-null: the certificate variant (fused register variants only)
    const int32_t *unit_list, *unit_count;   // non-null: only the listed units (blocks beyond the count exit)
    int routed_stride;                       // row stride of routed_pages (>= P)
    const uint16_t* tl_summaries;            // non-null: two-level front end (page_scores = representative scores)
    int P_super;
    cudaStream_t stream;
};


namespace {

template <int THREADS, int PAGE_KPT, int TOK_KPT, bool CERT>
cudaError_t launch_variant(const SparseArgs& a)
{
    static bool attr_done[kMaxDevices] = {};   // per template instance
    if (a.smem > 48 * 1024) {
        const cudaError_t e = allow_large_dynamic_smem(sparse_decode_kernel<THREADS, PAGE_KPT, TOK_KPT, CERT>, attr_done);
        if (e != cudaSuccess) return e;
    }
    const unsigned units = (unsigned)(a.g.batch * a.g.n_q_heads);
    return launch_pdl(sparse_decode_kernel<THREADS, PAGE_KPT, TOK_KPT, CERT>, dim3(units), dim3(THREADS), a.smem, a.stream,
                      a.g, a.q, a.k, a.v, a.block_table, a.seq_lens, a.routed_pages, a.page_scores, a.P, a.K_c, a.epsilon,
                      a.gap_threshold, a.out, a.diag, a.fallback_list, a.fallback_count, a.rad_logical, a.cert,
                      a.unit_list, a.unit_count, a.routed_stride, a.tl_summaries, a.P_super);
}

// token-score registers per thread from the number of routed tokens
template <int THREADS, int PAGE_KPT, bool CERT>
cudaError_t launch_tok(const SparseArgs& a)
{
    const int N = a.P * a.g.page_size;
    if (N <= 2 * THREADS) return launch_variant<THREADS, PAGE_KPT, 2, CERT>(a);
    if (N <= 4 * THREADS) return launch_variant<THREADS, PAGE_KPT, 4, CERT>(a);
    if constexpr (THREADS <= 256)
        return N <= 8 * THREADS ? launch_variant<THREADS, PAGE_KPT, 8, CERT>(a) : cudaErrorInvalidValue;
    else
        return cudaErrorInvalidValue;   // 128 pages * 16 tokens = 4 * 512: never reached
}

}  // namespace

// one variant per translation unit
cudaError_t launch_sparse_cert(const SparseArgs& a, int threads);        // routing certificate
cudaError_t launch_sparse_two_level(const SparseArgs& a, int threads);   // two-level front end

}  // namespace vsa
