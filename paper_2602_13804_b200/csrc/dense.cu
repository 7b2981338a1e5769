// Dense fallback (paper Sec. 10.3, "fallback-to-dense"): plain softmax attention over every token of
// the flagged units, as a split-K pass over the paged cache.
//
// This is the one place of the step where the arithmetic is a real dense contraction - the G query
// heads of a GQA group against the same K and V tiles - and where only the output (not a discrete
// decision) depends on it, so it runs on the tensor cores: per 16-token page and warp,
//   S[heads x 16]  = Q[heads x 128] . K_page^T      (16 mma.m16n8k16, bf16 in, fp32 accumulate)
//   O[heads x 128] += P[heads x 16] . V_page        (16 mma.m16n8k16)
// with the heads padded to the 16-row MMA tile and an online softmax in between.  K and V tiles
// stream through a per-warp cp.async ring (three pages deep, XOR-swizzled for ldmatrix).
//
// Work decomposition: an item is (sequence, KV head, range of pages); K and V are read once for all
// listed heads of the group.  The number of pages per item is chosen ON THE DEVICE from how much
// was flagged, so that one flagged head of a 128k-token sequence is spread over the whole chip
// while a full dense pass uses long items.  A persistent grid (one block per SM) walks the items;
// the block that finishes the last item of a (sequence, KV head) combines its partials.
#include <math.h>

#include <cuda.h>

#include "page_mma.cuh"
#include "vsa_device.cuh"
#include "vsa_launch.h"

namespace vsa {

namespace {

constexpr int kTileRows = 16;                      // the pass walks tiles of 16 tokens: one per 16-token page, two per 32-token page
constexpr int kPagesPerItemGoal = 128;             // pages per item and block from which a second round pays
constexpr int kMaxRounds = 2;
constexpr int kMaxRoundsRagged = 8;
constexpr float kPScale = 16384.0f;                // FP8: the probabilities' place in the f16 range

// Sizes that depend on the head dimension D (64, 128 or 256).  The ring of a block holds three stages of a
// K tile and a V tile per warp: 192 KB with eight warps at D = 128; D = 256 runs four warps per block so
// that the same ring fits.
// FP8 (D = 128): the unit of work is 32 tokens (two tiles); a stage holds their e4m3 rows as they are (4 KB of
// K, 4 KB of V), brought by four TMA tile loads in the 128-byte swizzle that ldmatrix wants; fragments are converted to f16
// (exact) for m16n8k16 MMAs with the tokens, then the columns, as rows and the heads as columns.
template <int D, bool FP8 = false>
struct DenseCfg {
    // fp8: a unit of half the bytes costs the same instructions per token, so the pass is bound by the latency of each
    // warp's chain: twelve warps with two stages.  Microseconds per layer, 16 sequences of 16k - 32k that all fall back
    // (754 MB), with 8 / 10 / 12 warps: 228 / 221 / 207.  Before, with m16n8k32 e4m3 MMAs of two terms per
    // operand (860 instructions per 32 tokens against 560 now) and 16-byte copies in place of TMA tiles, 290; a quarter of the
    // sequences (246 MB, the kernel alone 62 us, DRAM at half its rate, 0.40 of the issue slots) 116 -> 90.
    static constexpr int kDenseThreads = FP8 ? 384 : D == 256 ? 128 : 256;
    static constexpr int kStages = FP8 ? 2 : 3;                // units in flight per warp
    static constexpr int kDenseWarps = kDenseThreads / 32;
    static constexpr int kRowBytes = 2 * D;
    static constexpr int kTileBytes = kTileRows * kRowBytes;   // K (or V) rows of one tile and KV head (4 KB at D = 128)
    static constexpr int kUnitRows = FP8 ? 32 : kTileRows;     // tokens per unit of work of a warp
    static constexpr int kRawBytes = 32 * D;                   // FP8: K (or V) rows of a unit as e4m3 bytes
    static constexpr int kStageBytes = FP8 ? 2 * kRawBytes : 2 * kTileBytes;   // K + V
    static constexpr int kWarpBytes = kStages * kStageBytes;
    static constexpr int kRingBytes = kDenseWarps * kWarpBytes;
    static constexpr int kBarBytes = FP8 ? kDenseWarps * kStages * 8 : 0;   // one mbarrier per stage
    static constexpr int kPartialFloats = 2 + D;               // per (item, head): max (log2 domain), sum, acc[D]
    static constexpr int kMinPagesPerItem = 2 * kDenseWarps;   // at least two pages per warp: one would expose the DRAM latency
};

__device__ __forceinline__ void cp_async_16_zfill(uint32_t smem_addr, const void* gptr, bool valid)
{
    const int n = valid ? 16 : 0;   // src-size 0: the 16 destination bytes are zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr), "l"(gptr), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
// rows 8..15 of A are zero here
__device__ __forceinline__ void mma_bf16(float (&d)[4], uint32_t a0, uint32_t a2, uint32_t b0, uint32_t b1)
{
    mma_16816(d, a0, 0u, a2, 0u, b0, b1);
}
// D (16x8, fp32) += A (16x16, f16, row) * B (16x8, f16, col)
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                        uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// an 8 x 8 matrix of 16-bit elements, two of a row per lane, transposed across the warp
__device__ __forceinline__ uint32_t transpose_8x8(uint32_t x)
{
    uint32_t r;
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(x));
    return r;
}
// four e4m3 bytes as f16 (exact), bytes 0, 1 and bytes 2, 3
__device__ __forceinline__ void e4m3x4_to_f16(uint32_t bytes, uint32_t& lo, uint32_t& hi)
{
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tcvt.rn.f16x2.e4m3x2 %0, l;\n\tcvt.rn.f16x2.e4m3x2 %1, h;\n\t}"
        : "=r"(lo), "=r"(hi)
        : "r"(bytes));
}
__device__ __forceinline__ uint32_t pack_f16x2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// 16 x 16 bytes, transposed: lane (g = lane / 4, t = lane % 4) receives rows 4t .. 4t+3 of column g (first
// register) and of column g + 8 (second); .x2 loads a second matrix (addresses from lanes 16 .. 31) into r2, r3
__device__ __forceinline__ void ldmatrix_x2_trans_b8(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m16n16.x2.trans.shared.b8 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// one tile of 16 rows of 128 bytes: rows row .. row + 15 of KV head `head` of pool page `page`
__device__ __forceinline__ void tma_tile(uint32_t dst, const CUtensorMap* map, int row, int head, int page, uint32_t mbar)
{
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
                 ::"r"(dst), "l"(map), "r"(0), "r"(row), "r"(head), "r"(page), "r"(mbar)
                 : "memory");
}

// e4m3 cache: the K and V pools as tensors [page][head][token][128 bytes], box = one tile
template <bool FP8>
struct DenseMaps {};
template <>
struct DenseMaps<true> {
    CUtensorMap k, v;
};

struct DenseSmem {
    uint8_t* ring;         // [warps][stages][K tile | V tile]; reused for the cross-warp merge
    int32_t* item_base;    // [n_groups + 1] first item of every group (exclusive scan)
    uint8_t* group_mask;   // [n_groups] listed heads of the group
    int32_t* misc;         // [32]
};

// The partials of a (sequence, KV head) combined by the block that finished its last item.  Out of line: the kernel's
// registers and code are those of its main loop.
template <int G, int D, bool FP8>
__device__ __noinline__ void combine_items(float* ring, float* misc, const float* gp, int items_of_group, uint32_t mask,
                                           long long first_unit, float* out, vsa_diag_t* diag)
{
    using Cfg = DenseCfg<D, FP8>;
    constexpr int kDenseThreads = Cfg::kDenseThreads, kDenseWarps = Cfg::kDenseWarps, kPartialFloats = Cfg::kPartialFloats, kHeadDim = D;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // Every item's (max, sum) of every head in shared memory, then the listed heads and their items dealt out to the
    // warps: the loads are independent, and one head keeps every warp busy.  A thread per column that walked all
    // items paid a memory round trip for every eight of them: with this and the 32-bit divisions of the item sizes one
    // sequence of 128k that falls back 131 -> 118 us per layer, one unit of four in 4 of 2k - 8k 36.8 -> 34.5, the
    // same at D = 256 63.9 -> 56.4.
    float* ms_s = ring;                                 // [items][G]
    float* ls_s = ms_s + (size_t)items_of_group * G;    // [items][G]
    float* sums = ms_s + ((size_t)2 * items_of_group * G + 3) / 4 * 4;   // [warps][G][2 + D]
    for (int i = tid; i < items_of_group * G; i += kDenseThreads) {
        const float* rec = gp + (long long)i * kPartialFloats;
        ms_s[i] = __ldcg(rec);
        ls_s[i] = __ldcg(rec + 1);
    }
    __syncthreads();
    const int heads = __popc(mask), per_head = heads < kDenseWarps ? kDenseWarps / heads : 1;   // warps for each head
    const int slice = warp % per_head;
#pragma unroll 1
    for (int n = warp / per_head; n < heads; n += kDenseWarps / per_head) {
        uint32_t from_nth = mask;
        for (int i = 0; i < n; ++i) from_nth &= from_nth - 1u;
        const int hh = __ffs(from_nth) - 1;   // the n-th listed head
        float M = -INFINITY, failed = 0.0f;   // failed: -1 a page outside the pool, -2 a copy that did not land
        for (int it = lane; it < items_of_group; it += 32) {
            M = fmaxf(M, ms_s[it * G + hh]);
            failed = fminf(failed, ls_s[it * G + hh]);
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            M = fmaxf(M, __shfl_xor_sync(kFullMask, M, off));
            failed = fminf(failed, __shfl_xor_sync(kFullMask, failed, off));
        }
        constexpr int PAIRS = D / 64;   // columns 64 j + 2 lane, + 1
        float2 acc[PAIRS];
        float L = 0.0f;
#pragma unroll
        for (int j = 0; j < PAIRS; ++j) acc[j] = make_float2(0.0f, 0.0f);
#pragma unroll 4
        for (int it = slice; it < items_of_group; it += per_head) {
            const float ms = ms_s[it * G + hh];
            const float f = ms == -INFINITY ? 0.0f : exp2f(ms - M);
            const float2* rec = reinterpret_cast<const float2*>(gp + ((long long)it * G + hh) * kPartialFloats + 2) + lane;
#pragma unroll
            for (int j = 0; j < PAIRS; ++j) {
                const float2 x = __ldcg(rec + 32 * j);
                acc[j].x = fmaf(x.x, f, acc[j].x);
                acc[j].y = fmaf(x.y, f, acc[j].y);
            }
            L = fmaf(ls_s[it * G + hh], f, L);
        }
        float* mine = sums + (slice * G + hh) * kPartialFloats;
#pragma unroll
        for (int j = 0; j < PAIRS; ++j) reinterpret_cast<float2*>(mine + 2)[lane + 32 * j] = acc[j];
        if (lane == 0) mine[0] = L;
        if (lane == 0 && slice == 0) {
            misc[hh] = M;
            misc[16 + hh] = failed;
        }
    }
    __syncthreads();
    for (int idx = tid; idx < G * kHeadDim; idx += kDenseThreads) {
        const int hh = idx / kHeadDim, e = idx % kHeadDim;
        if (!((mask >> hh) & 1u)) continue;
        const long long unit = first_unit + hh;
        const float M = misc[hh], failed = misc[16 + hh];
        float acc = 0.0f, L = 0.0f;
        for (int w = 0; w < per_head; ++w) {
            const float* rec = sums + (w * G + hh) * kPartialFloats;
            acc += rec[2 + e];
            L += rec[0];
        }
        if (failed < 0.0f) {   // no dense result exists
            out[unit * kHeadDim + e] = 0.0f;
            if (e == 0 && diag) {
                diag[unit].lse = 0.0f;
                diag[unit].status = failed < -1.0f ? VSA_UNIT_COPY_TIMEOUT : VSA_UNIT_BAD_PAGE;
            }
            continue;
        }
        out[unit * kHeadDim + e] = L > 0.0f ? acc / L : 0.0f;
        if (e == 0 && diag) diag[unit].lse = (M + log2f(L)) * 0.6931471805599453f;
    }
}

template <int G, int D = vsa::kHeadDim, bool FP8 = false>
__global__ void __launch_bounds__((DenseCfg<D, FP8>::kDenseThreads), 1)
dense_split_kernel(Geometry geo, const uint16_t* __restrict__ q, const uint16_t* __restrict__ k_cache,
                   const uint16_t* __restrict__ v_cache, const int32_t* __restrict__ block_table,
                   const int32_t* __restrict__ seq_lens, int32_t* __restrict__ fallback_list,
                   int32_t* __restrict__ fallback_count, const int32_t* __restrict__ flags, float epsilon, float* __restrict__ partials,
                   int32_t* __restrict__ counters, float* __restrict__ out, vsa_diag_t* __restrict__ diag,
                   int max_items, const float* __restrict__ k_scale, const float* __restrict__ v_scale,
                   const __grid_constant__ DenseMaps<FP8> maps)
{
    static_assert(!FP8 || D == 128, "fp8 cache: head dimension 128");
    using Cfg = DenseCfg<D, FP8>;
    constexpr int kDenseThreads = Cfg::kDenseThreads, kDenseWarps = Cfg::kDenseWarps, kRowBytes = Cfg::kRowBytes,
                  kTileBytes = Cfg::kTileBytes, kStageBytes = Cfg::kStageBytes, kRingBytes = Cfg::kRingBytes,
                  kPartialFloats = Cfg::kPartialFloats, kStages = Cfg::kStages, kMinPagesPerItem = Cfg::kMinPagesPerItem, kHeadDim = D;
    constexpr int kUnit = Cfg::kUnitRows;
    constexpr int KS = D / 16;    // 16-element steps of the Q K^T contraction = 16-column steps of P V
    constexpr int NT = D / 8;     // 8-column output tiles
    constexpr int CPR = D / 8;    // 16-byte chunks per row
    constexpr int RPI = 32 / (CPR < 32 ? CPR : 32);   // rows one copy instruction of a warp covers
    extern __shared__ __align__(1024) uint8_t dense_smem[];   // (the TMA swizzle is one of address bits)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_groups = geo.batch * geo.n_kv_heads;
    DenseSmem sm;
    sm.ring = dense_smem;
    const uint32_t bars = (uint32_t)__cvta_generic_to_shared(dense_smem + kRingBytes);   // FP8: [warp][stage]
    sm.item_base = (int32_t*)(dense_smem + kRingBytes + Cfg::kBarBytes);
    sm.misc = sm.item_base + n_groups + 1;
    sm.group_mask = (uint8_t*)(sm.misc + 32);
    // The list is empty as a rule and the next kernel is what the stream waits for: that one may be scheduled while
    // this one still waits (0.3 us of a 15.5 us layer at batch 1).  Before its own wait it reads nothing that the
    // sparse pass, the only kernel it can then overlap, writes.
    pdl_launch_dependents();
    pdl_wait();
    if (!flags && fallback_count && ld_cg_s32(fallback_count) <= 0) return;   // the usual case: the shortest way

    // ---- which heads of which groups are listed? ----
    if (flags) {
        // one flag per unit (a step whose sparse pass ran the scan itself: nothing ahead of it could clear a counter); the
        // list is made here
        const int units = geo.batch * geo.n_q_heads;
        int mine = 0;
        for (int i = tid; i < units; i += kDenseThreads) mine |= __ldcg(flags + i);
        if (!__syncthreads_or(mine)) {
            if (blockIdx.x == 0 && tid == 0) *fallback_count = 0;
            return;
        }
        for (int i = tid; i < n_groups; i += kDenseThreads) sm.group_mask[i] = 0;
        if (tid == 0) sm.misc[31] = 0;
        __syncthreads();
        for (int i = tid; i < units; i += kDenseThreads) {
            if (__ldcg(flags + i) == 0) continue;
            const int grp = i / G;   // (heads of a group are neighbours)
            atomicOr(reinterpret_cast<unsigned int*>(sm.group_mask) + (grp >> 2), (1u << (i % G)) << (8 * (grp & 3)));
            if (blockIdx.x == 0) fallback_list[atomicAdd(&sm.misc[31], 1)] = i;
        }
        __syncthreads();
        if (blockIdx.x == 0 && tid == 0) *fallback_count = sm.misc[31];
        __syncthreads();
    } else if (fallback_count) {
        const int count = *fallback_count;
        for (int i = tid; i < n_groups; i += kDenseThreads) sm.group_mask[i] = 0;
        __syncthreads();
        for (int i = tid; i < count; i += kDenseThreads) {
            const int u = fallback_list[i];
            const int ub = u / geo.n_q_heads, uh = u % geo.n_q_heads;
            const int grp = ub * geo.n_kv_heads + uh / G;
            // byte-wide OR through the aligned 32-bit word that holds the group's byte
            atomicOr(reinterpret_cast<unsigned int*>(sm.group_mask) + (grp >> 2), (1u << (uh % G)) << (8 * (grp & 3)));
        }
    } else {
        for (int i = tid; i < n_groups; i += kDenseThreads) sm.group_mask[i] = (uint8_t)((1u << G) - 1u);
    }
    if (tid < 32) sm.misc[tid] = 0;
    if constexpr (FP8) {
        if (tid < kDenseWarps * kStages) mbar_init(bars + 8u * (uint32_t)tid, 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    // ---- pages per item from the amount of flagged work, then the item table ----
    int32_t* group_pages = reinterpret_cast<int32_t*>(sm.ring);   // (the ring is not in use yet; 16 KB at most)
    {
        int pages = 0, groups = 0, longest = 0;
        for (int i = tid; i < n_groups; i += kDenseThreads) {
            int p = 0;
            if (sm.group_mask[i]) {
                const int T = seq_lens[i / geo.n_kv_heads];
                if (geo.length_ok(T)) p = (T + kUnit - 1) / kUnit;
            }
            group_pages[i] = p;
            pages += p;
            groups += p > 0;
            longest = max(longest, p);
        }
#pragma unroll
        for (int off = 16; off; off >>= 1) {
            pages += __shfl_xor_sync(kFullMask, pages, off);
            groups += __shfl_xor_sync(kFullMask, groups, off);
            longest = max(longest, __shfl_xor_sync(kFullMask, longest, off));
        }
        if (lane == 0) {
            atomicAdd(&sm.misc[0], pages);
            atomicAdd(&sm.misc[1], groups);
            atomicMax(&sm.misc[2], longest);
        }
    }
    __syncthreads();
    const int total_pages = sm.misc[0], flagged_groups = sm.misc[1], longest_group = sm.misc[2];
    if (total_pages == 0) return;
    int ppi;   // pages per item, a multiple of the warp count
    {
        // Whole rounds: at most `rounds` items per block - one when the work is small (an item costs a few
        // microseconds of fixed overhead: query fragments, pipeline fill, merge, ticket), two when items
        // stay long.  Every group may add one ragged item, so sizing for (target - groups) full items
        // keeps the count within the target and no block starts a round the others do not have.
        // (32-bit divisions, which are a shorter chain; the counts are below 2^31)
        const unsigned blocks = gridDim.x, total = (unsigned)total_pages, listed = (unsigned)flagged_groups;
        unsigned rounds = total / (blocks * kPagesPerItemGoal);
        rounds = rounds < 1 ? 1 : (rounds > kMaxRounds ? kMaxRounds : rounds);   // 1 or 2
        // many flagged groups of uneven length (the longest more than twice the mean): about four items
        // per group, so that short and long groups mix over the blocks
        if ((long long)longest_group * flagged_groups > 2LL * total_pages) {
            const unsigned by_groups = (4 * listed + blocks - 1) / blocks;
            if (rounds < by_groups) rounds = by_groups < kMaxRoundsRagged ? by_groups : kMaxRoundsRagged;
        }
        const unsigned target = blocks * rounds, parts = target > 2 * listed ? target - listed : target;
        unsigned want = (total + parts - 1) / parts;
        const unsigned room = (unsigned)max_items - listed;
        const unsigned need = (total + room - 1) / room;
        if (want < need) want = need;
        ppi = (int)((want + kDenseWarps - 1) / kDenseWarps) * kDenseWarps;
        if (ppi < kMinPagesPerItem) ppi = kMinPagesPerItem;
    }
    {
        // exclusive scan of items per group: contiguous ranges per thread, then across threads
        const int per = (n_groups + kDenseThreads - 1) / kDenseThreads;
        const int lo = tid * per, hi = min(n_groups, lo + per);
        int mine = 0;
        for (int i = lo; i < hi; ++i) mine += (group_pages[i] + ppi - 1) / ppi;
        int incl = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(kFullMask, incl, off);
            if (lane >= off) incl += o;
        }
        if (lane == 31) sm.misc[16 + warp] = incl;
        __syncthreads();
        int base = incl - mine;
        for (int w = 0; w < warp; ++w) base += sm.misc[16 + w];
        for (int i = lo; i < hi; ++i) {
            sm.item_base[i] = base;
            base += (group_pages[i] + ppi - 1) / ppi;
        }
        if (tid == kDenseThreads - 1) sm.item_base[n_groups] = base;
    }
    if constexpr (FP8) fence_async_proxy();   // group_pages lay where the copies go
    __syncthreads();
    const int n_items = sm.item_base[n_groups];

    const float scale = 1.4426950408889634f / epsilon;   // scores are kept in the log2 domain
    const int head = lane >> 2;                          // MMA row of this lane = query head in the group
    const int quad = lane & 3;
    uint8_t* my_ring = sm.ring + warp * Cfg::kWarpBytes;
    const uint32_t ring_addr = (uint32_t)__cvta_generic_to_shared(my_ring);
    // copy mapping: lane covers 16-byte chunk lane % CPR of rows lane / CPR + RPI i, i = 0 .. 16 / RPI - 1
    const int cp_chunk = lane % CPR, cp_row0 = lane / CPR;
    int used = 0;   // FP8: units that this warp has asked for in earlier items

    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        // group of this item: last g with item_base[g] <= item
        int glo = 0, ghi = n_groups;
        while (ghi - glo > 1) {
            const int mid = (glo + ghi) >> 1;
            if (sm.item_base[mid] <= item) glo = mid; else ghi = mid;
        }
        const int grp = glo;
        const uint32_t mask = sm.group_mask[grp];
        const int b = grp / geo.n_kv_heads, g = grp % geo.n_kv_heads;
        const int T = seq_lens[b];
        const int nb = (T + kUnit - 1) / kUnit;   // units (tiles of 16 tokens; fp8: pairs of tiles) of the sequence
        const int chunk = item - sm.item_base[grp];
        const int items_of_group = sm.item_base[grp + 1] - sm.item_base[grp];
        // the group's pages are split evenly over its items (whole multiples of the warp count)
        const int even = ((nb + items_of_group - 1) / items_of_group + kDenseWarps - 1) / kDenseWarps * kDenseWarps;
        const int first_page = min(nb, chunk * even);
        const int end_page = min(nb, first_page + even);
        const int32_t* bt = block_table + (long long)b * geo.max_pages;

        float m_run = -INFINITY, l_run = 0.0f;   // per lane: head `head`, partial over this lane's columns
        float m_run1 = -INFINITY, l_run1 = 0.0f;   // FP8: of head 2 quad + 1 (m_run, l_run: of head 2 quad)
        constexpr int OT = FP8 ? D / 16 : NT;
        float o[OT][4];
#pragma unroll
        for (int n = 0; n < OT; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i) o[n][i] = 0.0f;

        // pages of this warp: first_page + warp, + 8, ...
        const int my_first = first_page + warp;
        const int my_count = my_first < end_page ? (end_page - my_first + kDenseWarps - 1) / kDenseWarps : 0;
        // fp8: the pool pages and the scales of 32 units at a time, one unit per lane (a page outside the pool fails the
        // group's listed heads); a table load in front of every unit's copies stalls the warp for a trip to L2.  (The bf16
        // pass sits at the HBM rate and lost 2 % to it.)  Tiles past the sequence and pages outside the pool are copied from
        // page 0, with scales of 0, and masked.
        int phys0 = 0, phys1 = 0;
        float kscale0 = 0.0f, kscale1 = 0.0f, vscale0 = 0.0f, vscale1 = 0.0f;
        auto look_up = [&](int k0) {
            const int pl = my_first + (k0 + lane) * kDenseWarps;
            auto entry = [&](int tile, float& ks, float& vs) {
                ks = vs = 0.0f;
                if (k0 + lane >= my_count || tile * kTileRows >= T) return 0;
                const int ph = bt[tile >> geo.tile_shift];
                if (ph < 0 || ph >= geo.pool_pages) {
                    atomicMax(&sm.misc[13], 1);   // (cleared at the end of the previous item)
                    return 0;
                }
                const long long at = (long long)ph * geo.kv_heads_stored + g / geo.kv_div;
                ks = k_scale[at];
                vs = v_scale[at];
                return ph;
            };
            phys0 = entry(2 * pl, kscale0, vscale0);
            phys1 = entry(2 * pl + 1, kscale1, vscale1);
            __syncwarp();
        };
        auto issue = [&](int k) {   // k-th unit of this warp into stage k % kStages
            if (FP8 && (k & 31) == 0) look_up(k);
            const int pl = my_first + k * kDenseWarps;
            if constexpr (FP8) {
                // four tiles of 2 KB, asked for by one lane (16 copies of 16 bytes per lane, with their addresses, took 116 us
                // per layer where the tiles took 108, all else the same)
                const int page0 = __shfl_sync(kFullMask, phys0, k & 31), page1 = __shfl_sync(kFullMask, phys1, k & 31);
                if (lane == 0) {
                    const int stage = (used + k) % kStages, in_page = (1 << geo.tile_shift) - 1, head_at = g / geo.kv_div;
                    const int row0 = ((2 * pl) & in_page) * kTileRows, row1 = ((2 * pl + 1) & in_page) * kTileRows;
                    const uint32_t dst = ring_addr + (uint32_t)(stage * kStageBytes);
                    const uint32_t bar = bars + 8u * (uint32_t)(warp * kStages + stage);
                    mbar_expect_tx(bar, kStageBytes);
                    tma_tile(dst, &maps.k, row0, head_at, page0, bar);
                    tma_tile(dst + Cfg::kRawBytes / 2, &maps.k, row1, head_at, page1, bar);
                    tma_tile(dst + Cfg::kRawBytes, &maps.v, row0, head_at, page0, bar);
                    tma_tile(dst + Cfg::kRawBytes * 3 / 2, &maps.v, row1, head_at, page1, bar);
                }
                __syncwarp();
            } else {
            const uint32_t dst = ring_addr + (uint32_t)((k % kStages) * kStageBytes);
            long long phys = bt[pl >> geo.tile_shift];
            const bool page_ok = phys >= 0 && phys < geo.pool_pages;
            if (!page_ok) {
                phys = 0;
                sm.misc[13] = 1;   // a page outside the pool: the group's listed heads fail (cleared after the item)
            }
            const int valid_rows = page_ok ? min(kTileRows, T - pl * kTileRows) : 0;
            const long long head_off = (long long)(g / geo.kv_div) * geo.head_stride + cp_chunk * 8 +
                                       (long long)((pl & ((1 << geo.tile_shift) - 1)) * kTileRows) * geo.token_stride;
            const uint16_t* kp = k_cache + phys * geo.page_stride + head_off;
            const uint16_t* vp = v_cache + phys * geo.page_stride + head_off;
#pragma unroll
            for (int i = 0; i < kTileRows / RPI; ++i) {
                const int r = cp_row0 + RPI * i;
                const uint32_t off = (uint32_t)(r * kRowBytes + ((cp_chunk ^ (r & 7)) << 4));
                const bool ok = r < valid_rows;
                cp_async_16_zfill(dst + off, kp + (long long)r * geo.token_stride, ok);
                cp_async_16_zfill(dst + kTileBytes + off, vp + (long long)r * geo.token_stride, ok);
            }
            }
        };
#pragma unroll
        for (int s = 0; s < kStages - 1; ++s) {
            if (s < my_count) issue(s);
            if constexpr (!FP8) cp_async_commit();
        }

        // Q fragments of the group, while the first tiles are on their way: bf16 pairs straight from memory, rows >= G are zero
        uint32_t qa0[KS], qa2[KS];
        float q_unscale = 1.0f;
        if constexpr (FP8) {
            // q as f16 operands, scaled by a power of two into the top of the f16 range: exact down to 2^-28 of the head's
            // largest element.  Step ks holds columns 16 ks + 4 quad, + 1 (qa0) and + 2, + 3 (qa2) of head lane / 4: the
            // order in which a lane receives the bytes of a key row.
            const uint16_t* qrow = q + ((long long)b * geo.n_q_heads + g * G + (head < G ? head : 0)) * kHeadDim;
            float qv[KS][4];
            float amax = 0.0f;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                const uint2 raw = *reinterpret_cast<const uint2*>(qrow + ks * 16 + quad * 4);
                qv[ks][0] = __uint_as_float(raw.x << 16);
                qv[ks][1] = __uint_as_float(raw.x & 0xffff0000u);
                qv[ks][2] = __uint_as_float(raw.y << 16);
                qv[ks][3] = __uint_as_float(raw.y & 0xffff0000u);
#pragma unroll
                for (int i = 0; i < 4; ++i) amax = fmaxf(amax, fabsf(qv[ks][i]));
            }
            amax = fmaxf(amax, __shfl_xor_sync(kFullMask, amax, 1));
            amax = fmaxf(amax, __shfl_xor_sync(kFullMask, amax, 2));
            const int sq = amax > 0.0f ? 13 - ilogbf(amax) : 0;   // largest |q| of the head lands in [2^13, 2^14)
            q_unscale = ldexpf(1.0f, -sq);
            const float up0 = ldexpf(1.0f, sq >> 1), up1 = ldexpf(1.0f, sq - (sq >> 1));   // 2^sq may be no float
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                const uint32_t v0 = pack_f16x2(qv[ks][0] * up0 * up1, qv[ks][1] * up0 * up1);
                const uint32_t v2 = pack_f16x2(qv[ks][2] * up0 * up1, qv[ks][3] * up0 * up1);
                qa0[ks] = head < G ? v0 : 0u;
                qa2[ks] = head < G ? v2 : 0u;
            }
        } else {
            const uint16_t* qrow = q + ((long long)b * geo.n_q_heads + g * G + (head < G ? head : 0)) * kHeadDim;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                const uint32_t v0 = *reinterpret_cast<const uint32_t*>(qrow + ks * 16 + quad * 2);
                const uint32_t v2 = *reinterpret_cast<const uint32_t*>(qrow + ks * 16 + 8 + quad * 2);
                qa0[ks] = head < G ? v0 : 0u;
                qa2[ks] = head < G ? v2 : 0u;
            }
        }
        // FP8: the lane's score columns are heads 2 quad, 2 quad + 1; o[n]: columns 16 n + head and + 8 of both
        const float q_unscale0 = FP8 ? __shfl_sync(kFullMask, q_unscale, 8 * quad) * scale : 0.0f;
        const float q_unscale1 = FP8 ? __shfl_sync(kFullMask, q_unscale, 8 * quad + 4) * scale : 0.0f;
        for (int k = 0; k < my_count; ++k) {
            float ks0 = 0.0f, ks1 = 0.0f, vs0 = 0.0f, vs1 = 0.0f;
            if constexpr (FP8) {   // (before the next look-up)
                static_assert(kStages == 2, "a look-up is one unit ahead at most");
                ks0 = __shfl_sync(kFullMask, kscale0, k & 31), ks1 = __shfl_sync(kFullMask, kscale1, k & 31);
                vs0 = __shfl_sync(kFullMask, vscale0, k & 31), vs1 = __shfl_sync(kFullMask, vscale1, k & 31);
            }
            if (k + kStages - 1 < my_count) issue(k + kStages - 1);
            if constexpr (FP8) {
                const int seq = used + k;
                const uint32_t bar = bars + 8u * (uint32_t)(warp * kStages + seq % kStages);
                // (waited for once more before the stage can be written again or the block can end)
                if (!mbar_wait(bar, (uint32_t)(seq / kStages) & 1u)) {
                    atomicMax(&sm.misc[13], 2);
                    mbar_wait(bar, (uint32_t)(seq / kStages) & 1u);
                }
            } else {
                cp_async_commit();
                cp_async_wait<kStages - 1>();
            }
            __syncwarp();
            if constexpr (FP8) {
            const int pl = my_first + k * kDenseWarps;
            const int valid = min(kUnit, T - pl * kUnit);   // > 0
            const int stage = (used + k) % kStages;
            const uint32_t kbase = ring_addr + (uint32_t)(stage * kStageBytes);
            const uint32_t vbase = kbase + Cfg::kRawBytes;
            if (valid < kUnit) {   // value rows past the sequence have weight 0, but may hold NaN
                uint4* row = reinterpret_cast<uint4*>(my_ring + stage * kStageBytes + Cfg::kRawBytes + lane * 128);
                if (lane >= valid)
#pragma unroll
                    for (int i = 0; i < 8; ++i) row[i] = make_uint4(0u, 0u, 0u, 0u);
                __syncwarp();
            }

            // S^T = K Q^T for the 32 tokens of the unit (two 16-token row tiles): tokens are the rows of the MMA, which the
            // few heads of a group would leave half empty
            float st[2][4];
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int i = 0; i < 4; ++i) st[j][i] = 0.0f;
            {
                // ldmatrix.x4 on byte rows: matrix mi = lane / 8 is (tokens 8 (mi / 2) .. + 7) x (16-byte chunk 2 ks + mi % 2);
                // a lane receives 4 consecutive columns of one token: two slots of either half of a step, see qa0
                const int mi = lane >> 3, rr = lane & 7;
#pragma unroll
                for (int ks = 0; ks < 4; ++ks)
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        const int tok = hf * 16 + (mi >> 1) * 8 + rr, ch = 2 * ks + (mi & 1);
                        uint32_t r[4], a[4];
                        ldmatrix_x4(r, kbase + (uint32_t)(tok * 128 + ((ch ^ (tok & 7)) << 4)));
#pragma unroll
                        for (int i = 0; i < 2; ++i) {
                            e4m3x4_to_f16(r[i], a[0], a[2]);
                            e4m3x4_to_f16(r[2 + i], a[1], a[3]);
                            mma_f16(st[hf], a[0], a[1], a[2], a[3], qa0[2 * ks + i], qa2[2 * ks + i]);
                        }
                    }
            }
            // this lane: heads 2 quad (ta) and 2 quad + 1 (tb), tokens head + 8 j (head = lane / 4)
            float ta[4], tb[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {   // the page's key scale folded in
                ta[j] = st[j >> 1][2 * (j & 1)] * (q_unscale0 * (j < 2 ? ks0 : ks1));
                tb[j] = st[j >> 1][2 * (j & 1) + 1] * (q_unscale1 * (j < 2 ? ks0 : ks1));
            }
            if (valid < kUnit)
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (head + 8 * j >= valid) ta[j] = tb[j] = -INFINITY;
            float ma = fmaxf(fmaxf(ta[0], ta[1]), fmaxf(ta[2], ta[3])), mb = fmaxf(fmaxf(tb[0], tb[1]), fmaxf(tb[2], tb[3]));
            // a new maximum, rarer with every unit: reduce it and rescale the sums
            if (__any_sync(kFullMask, ma > m_run || mb > m_run1)) {
#pragma unroll
                for (int off = 4; off < 32; off <<= 1) {
                    ma = fmaxf(ma, __shfl_xor_sync(kFullMask, ma, off));
                    mb = fmaxf(mb, __shfl_xor_sync(kFullMask, mb, off));
                }
                ma = fmaxf(ma, m_run), mb = fmaxf(mb, m_run1);   // finite: token 0 of a unit is always valid
                const float fa = exp2f(m_run - ma), fb = exp2f(m_run1 - mb);   // 0 on the first unit
                l_run *= fa, l_run1 *= fb;
#pragma unroll
                for (int n = 0; n < OT; ++n) {
                    o[n][0] *= fa, o[n][1] *= fb;
                    o[n][2] *= fa, o[n][3] *= fb;
                }
                m_run = ma, m_run1 = mb;
            }
            // P as f16 operands: p * kPScale, normal numbers down to p = 2^-28; packed by token, then transposed into the B
            // fragment (tokens are the contraction's index)
            uint32_t pb[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float pa = exp2f(ta[j] - m_run), pc = exp2f(tb[j] - m_run1);
                l_run += pa, l_run1 += pc;
                pb[j] = transpose_8x8(pack_f16x2(pa * kPScale, pc * kPScale));
            }

            // O^T += V^T P^T, 16 columns at a time: one transposing byte load per 32 tokens x 16 columns.  A lane's four rows
            // of a column are tokens 2 quad, 2 quad + 1, 8 + 2 quad, 9 + 2 quad of the half: two slots of either half of a step.
            {
                const int rrow = lane & 15, qd = rrow >> 2, ii = rrow & 3;
                const int tokp = (lane >> 4) * 16 + ((ii < 2) ? 0 : 8) + 2 * qd + (ii & 1);
                const uint32_t vrow = vbase + (uint32_t)(tokp * 128);
                const float out0 = vs0 * (1.0f / kPScale), out1 = vs1 * (1.0f / kPScale);
#pragma unroll
                for (int dp = 0; dp < 8; ++dp) {
                    uint32_t r[4], a[4];
                    ldmatrix_x2_trans_b8(r, vrow + (uint32_t)((dp ^ (tokp & 7)) << 4));
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        float t[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                        e4m3x4_to_f16(r[2 * hf], a[0], a[2]);
                        e4m3x4_to_f16(r[2 * hf + 1], a[1], a[3]);
                        mma_f16(t, a[0], a[1], a[2], a[3], pb[2 * hf], pb[2 * hf + 1]);
#pragma unroll
                        for (int i = 0; i < 4; i += 2)
                            fma2(o[dp][i], o[dp][i + 1], t[i], t[i + 1], hf ? out1 : out0, hf ? out1 : out0);
                    }
                }
            }
            } else {
            const int pl = my_first + k * kDenseWarps;
            const int valid = min(kTileRows, T - pl * kTileRows);   // > 0
            const uint32_t kbase = ring_addr + (uint32_t)((k % kStages) * kStageBytes);
            const uint32_t vbase = kbase + kTileBytes;

            // S = Q K^T for the 16 tokens of the page (two 8-token column tiles)
            float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
            {
                const int mi = lane >> 3, tok = (mi >> 1) * 8 + (lane & 7);
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) {
                    const int ch = 2 * ks + (mi & 1);
                    uint32_t r[4];
                    ldmatrix_x4(r, kbase + (uint32_t)(tok * kRowBytes + ((ch ^ (tok & 7)) << 4)));
                    mma_bf16(s0, qa0[ks], qa2[ks], r[0], r[1]);
                    mma_bf16(s1, qa0[ks], qa2[ks], r[2], r[3]);
                }
            }
            // this lane: head `head`, tokens 2 quad, 2 quad + 1 (tile 0) and 8 + the same (tile 1)
            const float tscale = scale;
            float t[4];
            t[0] = (2 * quad < valid) ? s0[0] * tscale : -INFINITY;
            t[1] = (2 * quad + 1 < valid) ? s0[1] * tscale : -INFINITY;
            t[2] = (8 + 2 * quad < valid) ? s1[0] * tscale : -INFINITY;
            t[3] = (8 + 2 * quad + 1 < valid) ? s1[1] * tscale : -INFINITY;
            float pm = fmaxf(fmaxf(t[0], t[1]), fmaxf(t[2], t[3]));
            pm = fmaxf(pm, __shfl_xor_sync(kFullMask, pm, 1));
            pm = fmaxf(pm, __shfl_xor_sync(kFullMask, pm, 2));
            const float m_new = fmaxf(m_run, pm);       // finite: token 0 of a page is always valid
            const float corr = exp2f(m_run - m_new);    // 0 on the first page
            float p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) p[i] = exp2f(t[i] - m_new);
            l_run = fmaf(l_run, corr, (p[0] + p[1]) + (p[2] + p[3]));
            if (__any_sync(kFullMask, m_new > m_run)) {
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    o[n][0] *= corr;
                    o[n][1] *= corr;
                }
            }
            m_run = m_new;
            const uint32_t pa0 = pack_bf16x2(p[0], p[1]), pa2 = pack_bf16x2(p[2], p[3]);

            // O += P V
            {
                const int mi = lane >> 3, tok = (mi & 1) * 8 + (lane & 7);
#pragma unroll
                for (int dp = 0; dp < KS; ++dp) {
                    const int ch = 2 * dp + (mi >> 1);
                    uint32_t r[4];
                    ldmatrix_x4_trans(r, vbase + (uint32_t)(tok * kRowBytes + ((ch ^ (tok & 7)) << 4)));
                    mma_bf16(o[2 * dp], pa0, pa2, r[0], r[1]);
                    mma_bf16(o[2 * dp + 1], pa0, pa2, r[2], r[3]);
                }
            }
            }
            __syncwarp();   // the stage is overwritten by a later issue
        }
        if constexpr (FP8)
            used += my_count;   // (every one of them has been waited for)
        else
            cp_async_wait<0>();

        // ---- merge: the lanes that share a head (sum l), then the warps, into one partial per head ----
        float* mg = reinterpret_cast<float*>(sm.ring);   // [warps][G][2 + 128], in the place of the ring
        if constexpr (FP8) {
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) {
                l_run += __shfl_xor_sync(kFullMask, l_run, off);
                l_run1 += __shfl_xor_sync(kFullMask, l_run1, off);
            }
            __syncthreads();   // every warp is done with its ring
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int hh = 2 * quad + i;
                if (hh >= G) continue;
                float* rec = mg + (warp * G + hh) * kPartialFloats;
                if (head == 0) {
                    rec[0] = i ? m_run1 : m_run;
                    rec[1] = i ? l_run1 : l_run;
                }
#pragma unroll
                for (int n = 0; n < OT; ++n) {
                    rec[2 + n * 16 + head] = o[n][i];
                    rec[2 + n * 16 + 8 + head] = o[n][2 + i];
                }
            }
        } else {
            l_run += __shfl_xor_sync(kFullMask, l_run, 1);
            l_run += __shfl_xor_sync(kFullMask, l_run, 2);
            __syncthreads();   // every warp is done with its ring
            if (head < G) {
                float* rec = mg + (warp * G + head) * kPartialFloats;
                if (quad == 0) {
                    rec[0] = m_run;
                    rec[1] = l_run;
                }
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    rec[2 + n * 8 + quad * 2] = o[n][0];
                    rec[2 + n * 8 + quad * 2 + 1] = o[n][1];
                }
            }
        }
        __syncthreads();
        for (int idx = tid; idx < G * kHeadDim; idx += kDenseThreads) {
            const int hh = idx / kHeadDim, e = idx % kHeadDim;
            if (!((mask >> hh) & 1u)) continue;
            float M = -INFINITY;
#pragma unroll
            for (int w = 0; w < kDenseWarps; ++w) M = fmaxf(M, mg[(w * G + hh) * kPartialFloats]);
            float a = 0.0f, L = 0.0f;
#pragma unroll
            for (int w = 0; w < kDenseWarps; ++w) {
                const float* rec = mg + (w * G + hh) * kPartialFloats;
                const float f = rec[0] == -INFINITY ? 0.0f : exp2f(rec[0] - M);
                a = fmaf(rec[2 + e], f, a);
                L = fmaf(rec[1], f, L);
            }
            float* dst = partials + ((long long)item * G + hh) * kPartialFloats;
            dst[2 + e] = a;
            if (e == 0) {
                dst[0] = M;
                // sums are never negative: -1 marks a page outside the pool, -2 a copy that did not land
                dst[1] = sm.misc[13] ? -(float)sm.misc[13] : L;
            }
        }

        // ---- the block that finishes the last item of this (sequence, KV head) combines them ----
        __syncthreads();
        if (tid == 0) {
            __threadfence();   // (cumulative over the barrier)
            const bool last = atomicAdd(&counters[grp], 1) == items_of_group - 1;
            if (last) __threadfence();
            sm.misc[12] = last;
        }
        __syncthreads();
        if (sm.misc[12]) {
            combine_items<G, D, FP8>(reinterpret_cast<float*>(sm.ring), reinterpret_cast<float*>(sm.misc),
                                     partials + (long long)sm.item_base[grp] * G * kPartialFloats, items_of_group, mask,
                                     (long long)b * geo.n_q_heads + g * G, out, diag);
        }
        if (tid == 0) sm.misc[13] = 0;
        if constexpr (FP8) fence_async_proxy();
        __syncthreads();   // the ring (merge buffer) and misc are reused by the next item
    }
}

int num_sms() { return device_sm_count(); }

// room for the items the kernel may create: one ragged item per group plus the balancing target
int dense_max_items(const Geometry& g) { return g.batch * g.n_kv_heads + 2048; }

size_t dense_smem_bytes(const Geometry& g, bool fp8 = false)
{
    const size_t n_groups = (size_t)g.batch * g.n_kv_heads;
    const size_t ring = fp8 ? DenseCfg<128, true>::kRingBytes + DenseCfg<128, true>::kBarBytes
                            : g.head_dim == 64 ? DenseCfg<64>::kRingBytes
                                               : (g.head_dim == 256 ? DenseCfg<256>::kRingBytes : DenseCfg<128>::kRingBytes);
    return ring + (n_groups + 1) * 4 + 32 * 4 + (n_groups + 15) / 16 * 16;
}

}  // namespace

// A pool of e4m3 rows as a 4-d tensor, box = one tile of 16 rows, swizzled as ldmatrix reads it.  The entry points have
// checked what the encoding asks for: base and strides are multiples of 16 bytes.  (The stride of an extent of one page or
// head is never used; it may be any number.)
static bool encode_pool(CUtensorMap* map, const void* pool, const Geometry& g)
{
    using Encode = decltype(&cuTensorMapEncodeTiled);
    static const Encode encode = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult found;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &found) != cudaSuccess ||
            found != cudaDriverEntryPointSuccess)
            f = nullptr;
        return reinterpret_cast<Encode>(f);
    }();
    if (!encode) return false;
    const cuuint64_t dims[4] = {128, (cuuint64_t)g.page_size, (cuuint64_t)g.kv_heads_stored, (cuuint64_t)g.pool_pages};
    const cuuint64_t strides[3] = {(cuuint64_t)g.token_stride, (cuuint64_t)(g.kv_heads_stored > 1 ? g.head_stride : 128),
                                   (cuuint64_t)(g.pool_pages > 1 ? g.page_stride : 128)};
    const cuuint32_t box[4] = {128, kTileRows, 1, 1}, element_strides[4] = {1, 1, 1, 1};
    return encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(pool), dims, strides, box, element_strides,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static size_t dense_counter_bytes(const Geometry& g_in)
{
    const Geometry g = with_virtual_kv_heads(g_in);
    return (((size_t)g.batch * g.n_kv_heads * sizeof(int32_t)) + 255) / 256 * 256;
}

int32_t* dense_tickets(void* ws_dense) { return (int32_t*)ws_dense; }

int dense_ticket_count(const Geometry& g_in)
{
    const Geometry g = with_virtual_kv_heads(g_in);
    return g.batch * g.n_kv_heads;
}

size_t dense_workspace_bytes(const Geometry& g_in)
{
    const Geometry g = with_virtual_kv_heads(g_in);
    return dense_counter_bytes(g) + (size_t)dense_max_items(g) * g.group * (2 + g.head_dim) * sizeof(float);
}

void* dense_partials(const Geometry& g, void* ws_dense) { return (char*)ws_dense + dense_counter_bytes(g); }

size_t dense_partials_bytes(const Geometry& g) { return dense_workspace_bytes(g) - dense_counter_bytes(g); }

template <int G, int D, bool FP8 = false>
static cudaError_t launch_dense_gd(const Geometry& g, const uint16_t* q, const uint16_t* k, const uint16_t* v,
                                   const int32_t* block_table, const int32_t* seq_lens, int32_t* fallback_list,
                                   int32_t* fallback_count, const int32_t* flags, float epsilon, float* partials, int32_t* counters,
                                   float* out, vsa_diag_t* diag, cudaStream_t stream, const float* k_scale = nullptr,
                                   const float* v_scale = nullptr)
{
    const size_t smem = dense_smem_bytes(g, FP8);
    static bool attr_done[kMaxDevices] = {};   // per template instance
    const cudaError_t e = allow_large_dynamic_smem(dense_split_kernel<G, D, FP8>, attr_done);
    if (e != cudaSuccess) return e;
    DenseMaps<FP8> maps;
    if constexpr (FP8)
        if (!encode_pool(&maps.k, k, g) || !encode_pool(&maps.v, v, g)) return cudaErrorInvalidValue;
    // persistent grid: one block per SM (the ring fills the shared memory)
    return launch_pdl(dense_split_kernel<G, D, FP8>, dim3((unsigned)num_sms()), dim3(DenseCfg<D, FP8>::kDenseThreads), smem,
                      stream, g, q, k, v, block_table, seq_lens, fallback_list, fallback_count, flags, epsilon, partials,
                      counters, out, diag, dense_max_items(g), k_scale, v_scale, maps);
}

template <int G>
static cudaError_t launch_dense_g(const Geometry& g, const uint16_t* q, const uint16_t* k, const uint16_t* v,
                                  const int32_t* block_table, const int32_t* seq_lens, int32_t* fallback_list,
                                  int32_t* fallback_count, const int32_t* flags, float epsilon, float* partials, int32_t* counters,
                                  float* out, vsa_diag_t* diag, cudaStream_t stream, const float* k_scale,
                                  const float* v_scale)
{
    if (k_scale)
        return launch_dense_gd<G, 128, true>(g, q, k, v, block_table, seq_lens, fallback_list, fallback_count, flags, epsilon,
                                             partials, counters, out, diag, stream, k_scale, v_scale);
    if (g.head_dim == 64)
        return launch_dense_gd<G, 64>(g, q, k, v, block_table, seq_lens, fallback_list, fallback_count, flags, epsilon,
                                      partials, counters, out, diag, stream);
    if (g.head_dim == 256)
        return launch_dense_gd<G, 256>(g, q, k, v, block_table, seq_lens, fallback_list, fallback_count, flags, epsilon,
                                       partials, counters, out, diag, stream);
    return launch_dense_gd<G, 128>(g, q, k, v, block_table, seq_lens, fallback_list, fallback_count, flags, epsilon, partials,
                                   counters, out, diag, stream);
}

cudaError_t launch_dense(const Geometry& g_in, const void* q, const void* k_cache, const void* v_cache,
                         const int32_t* block_table, const int32_t* seq_lens, const int32_t* fallback_list_in,
                         const int32_t* fallback_count_in, float epsilon, float* out, vsa_diag_t* diag, void* ws,
                         cudaStream_t stream, bool tickets_cleared, const float* k_scale, const float* v_scale, const int32_t* flags)
{
    if ((k_scale || v_scale) && (!k_scale || !v_scale || g_in.head_dim != kHeadDim)) return cudaErrorInvalidValue;
    const Geometry g = with_virtual_kv_heads(g_in);
    int32_t *fallback_list = const_cast<int32_t*>(fallback_list_in), *fallback_count = const_cast<int32_t*>(fallback_count_in);   // (written with flags only)
    int32_t* counters = (int32_t*)ws;
    float* partials = (float*)dense_partials(g, ws);
    if (!tickets_cleared) {
        cudaError_t e = cudaMemsetAsync(counters, 0, dense_counter_bytes(g), stream);
        if (e != cudaSuccess) return e;
    }
    const uint16_t *qq = (const uint16_t*)q, *kk = (const uint16_t*)k_cache, *vv = (const uint16_t*)v_cache;
    switch (g.group) {
        case 1: return launch_dense_g<1>(g, qq, kk, vv, block_table, seq_lens, fallback_list, fallback_count, flags, epsilon, partials, counters, out, diag, stream, k_scale, v_scale);
        case 2: return launch_dense_g<2>(g, qq, kk, vv, block_table, seq_lens, fallback_list, fallback_count, flags, epsilon, partials, counters, out, diag, stream, k_scale, v_scale);
        case 4: return launch_dense_g<4>(g, qq, kk, vv, block_table, seq_lens, fallback_list, fallback_count, flags, epsilon, partials, counters, out, diag, stream, k_scale, v_scale);
        case 8: return launch_dense_g<8>(g, qq, kk, vv, block_table, seq_lens, fallback_list, fallback_count, flags, epsilon, partials, counters, out, diag, stream, k_scale, v_scale);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace vsa
