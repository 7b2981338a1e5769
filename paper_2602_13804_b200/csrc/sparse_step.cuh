// Fused sparse pass of one (sequence, query head) unit per thread block (paper Sec. 7 steps 2-4, Sec. 8 gap
// statistic, Cor. 1 leakage bound, Sec. 10.3 fallback flag):
//   [top-P page selection from the page scores] -> score every valid token of the routed pages -> exact
//   top-K_c -> weights -> weighted sum of the candidates' value rows -> diagnostics.
//
// A unit is a chain of short dependent phases, so what it costs is the number of instructions and block
// barriers on its longest thread and, since every instruction is executed once or twice per launch, the size
// of the code (instruction fetch: an SM caches about 2000 instructions, straight code that is not there takes three or more
// cycles each).  Hence: loops that run from memory instead of unrolled register arrays, one template instance for every
// table width, P and K_c, the rare exact fallbacks out of line, one barrier between phases.
//   * Page scores are staged in shared memory (16-byte copies, any table width).  In every warp the r-th largest
//     of the lanes' maxima, r = ceil(P / warps), has r scores at or above it; the smallest of these over the warps
//     bounds the P-th best score from below and leaves about 1.6 P scores, which are listed and ranked exactly.
//   * Ties are decided by (key << 32) | ~position.
//   * A warp that scored a tile keeps its keys in shared memory and selects among them; the candidates of all warps
//     are then compacted into one list, whose value rows are dealt out evenly to the groups of lanes.
//   * Every score is a chain of mixed-precision FMAs on the packed bf16 words (no unpacking).
// Measured, microseconds per layer before (register-array kernel with seventeen barriers) and after: 15.1 -> 13.1
// at batch 1, T = 4k with the scan and the empty dense pass; 21.2 -> 17.9 at T = 128k; batch 8, T = 32k 24.6 -> 23.3;
// 64 sequences of 4k - 128k with 8 heads a group 449 -> 399; batch 32 of short rows at D = 64 44 -> 39.  Then, with bulk
// copies of the key tiles and the value rows streamed through shared memory (128 threads), 355 -> 312 for the 64 sequences and
// 83.0 -> 81.5 at batch 16, T = 128k; with scores in registers where a thread has one chunk (and the append's reads side by
// side), 14.4 -> 14.2 at batch 1, T = 4k, the append included.
// What bounds it:
// no unit of the SM, but the chain of phases, until there are units enough to fill one another's waits.  Counters at P = 32, K_c = 256: 20k
// warp instructions per unit of 256 threads and 10k for the scan of its cluster, 0.40 of the issue slots at two units per SM (256
// units, 32k); 16k at four units of 128 threads, 0.45 (512 units of 8k); at P = 64, K_c = 512 35k, 0.62 at five (2048 units).  The waits are for
// the results of instructions, for shared memory and for loads from L2, in this order.
#pragma once

#include <limits.h>
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "page_mma.cuh"
#include "step_solve.cuh"
#include "vsa_device.cuh"
#include "vsa_launch.h"
#include "vsa_team.cuh"

namespace vsa {

// Shared-memory layout in 4-byte words, see step_layout.
struct StepLayout {
    int hist, warp_stat, misc, win_key, list, tokens, zeroed /* words from 0 cleared at the start */, win, loc, tile_off, tile_pos, tile_phys, keys, red, zred, bar, cand, solve, work, vring, bt, scan_q, scan_ring;
    int total;
    bool stage_bt;   // the block-table row is copied before the wait (blocks that wait for the scan anyway)
};

// Everything one launch needs.
struct StepParams {
    Geometry geo;
    StepLayout lay;
    int group_shift;            // log2(query heads per KV head)
    const uint16_t *q, *k, *v;
    const int32_t *block_table, *seq_lens;
    int32_t* routed_pages;
    const float* page_scores;   // nullptr: routed_pages is an input, or (summaries) the scores are computed here
    const uint16_t* summaries;  // without page_scores: the page scan runs here, by a cluster of the blocks of a KV head's query heads
    const uint32_t* bounds;     // not nullptr: page_scores are within page_score_slack() / 2 of the fixed-order ones, see route_mma.cu
    int cluster_shift;          // log2(blocks of a cluster): those of the heads, the first of them, and others that only scan
    int heads_shift;            // log2(heads of a cluster)
    int scan_per_sm;            // blocks of such a launch that share an SM
    bool scan_mma;              // scores by MMAs (page_mma.cuh)
    int* active_clusters;       // not nullptr: no launch, but active_clusters() of it
    bool by_position;           // tiles in the order of positions instead of scores (see BY_POSITION)
    int32_t* flags;             // with summaries: fallback flag of every unit, from which the dense pass makes the list
    int32_t* tickets;           // with summaries: the dense pass's tickets, cleared here
    int n_tickets;
    int P, K_c;
    float epsilon, gap_threshold;
    float* out;
    vsa_diag_t* diag;
    int32_t *fallback_list, *fallback_count;
    int solver_iters;
    vsa_solve_t* solve;
    const float *k_scale, *v_scale;   // fp8 cache
};

// one family of instances per translation unit
cudaError_t launch_step(const StepParams& p, int threads, cudaStream_t stream);        // head dimension 128
cudaError_t launch_step_d64(const StepParams& p, int threads, cudaStream_t stream);
cudaError_t launch_step_d256(const StepParams& p, int threads, cudaStream_t stream);
cudaError_t launch_step_fp8(const StepParams& p, int threads, cudaStream_t stream);    // e4m3 cache
cudaError_t launch_step_solve(const StepParams& p, int kind, cudaStream_t stream);     // iterative solves, 256 threads

namespace {

constexpr int kStepPages = 512;   // entries of the page list
constexpr int kStepList = 256;    // entries of the cut bucket's list
constexpr int kMaxRouted = 128;   // routed pages of a unit at most
constexpr int kStepBins = 256;    // histogram bins of the token selection
// iterative solve: scores and positions of the candidates, weights exchanged inside a warp, the readout
constexpr int kSolveWords = 3 * VSA_SOLVER_MAX_CANDIDATES + kHeadDim;
// control words
enum : int {
    kCtlStat = 0,       // 4 words, see publish below
    kCtlPages = 4,      // listed pages
    kCtlTokens,         // listed tokens of the cut bucket
    kCtlOut,            // key of the best rejected token
    kCtlBad,            // a routed page has no valid pool page
    kCtlMissing,        // tokens the last page lacks, once per time it is routed
    kCtlNp,             // routed pages (when they are an input)
    kCtlLate,           // a tile's copy did not arrive
    kCtlNext,           // key of the best page that is not routed
    kCtlCut,            // (tokens above the cut bucket << 20) | (tokens inside << 8) | bucket
    kCtlNear = 16,      // 4 words: bit t, the scores of the pages of rank t and t + 1 are too close to tell (P is 128 at most)
    kCtlBound = 20,     // bits of the largest sum |q_i k_i| of the pages (scan by the cluster)
    kCtlWords = 24
};

__host__ __device__ constexpr int step_lanes_per_row(int D) { return D / 8; }
// Value rows in flight per group of lanes, in stages of four in shared memory (0: in registers, see the value gather).  An
// iterative solve asks for all of its rows at once (16 per group at most), in the place of its key tile.
__host__ __device__ constexpr int step_value_stages(int threads, bool solve)
{
    return solve ? 4 : threads == 128 ? 2 : threads == 256 ? 3 : 0;
}

// Tiles of 16 summary rows in flight per warp of a scanning block: 8 KB.
__host__ __device__ constexpr int step_scan_stages(int D) { return D == 64 ? 4 : D == 128 ? 2 : 1; }

// Blocks whose tiles may come in either order, see BY_POSITION
__host__ __device__ constexpr bool step_order_open(int threads, int D, bool fp8) { return !fp8 && (threads == 512 || (threads == 128 && D == 64)); }

// near: page scores by MMAs, whose near ties are settled.  line: words that the parts which rows pass through start on a multiple of
inline StepLayout step_layout_on(int line, int threads, int D, int max_pages, int P, int PT, int K_c, bool fused, bool fp8, bool solve,
                              int cluster, int heads, bool near)
{
    StepLayout s;
    auto up = [&](int words) { return (words + line - 1) / line * line; };
    const int groups = threads / step_lanes_per_row(D), warps = threads / 32;
    const int tt = (PT + groups - 1) / groups;   // tiles of a group of lanes
    const int cands = (K_c + 4 * groups - 1) / (4 * groups) * (4 * groups);   // (the value gather takes four rows per group at a time)
    const int lane_words = fp8 ? 2 : 4;          // a lane's piece of a row
    const int keys = tt * groups * 16 * (D == 256 ? 2 : 1);   // [round][sub][thread]
    int o = up(kCtlWords);
    s.hist = o, o += kStepBins;
    s.tokens = o, o += 2 * kStepList;
    s.list = o;
    s.zeroed = s.list + 2 * kStepPages;
    s.keys = o;   // the page list is dead when the first token key is written
    o += keys > 2 * kStepPages ? keys : 2 * kStepPages;
    s.warp_stat = o, o += 2 * 16;
    s.misc = o, o += 16;
    s.win = o, o += (P + 15) & ~15;
    s.win_key = o, o += near ? 2 * ((P + 3) & ~3) : 0;   // and those of the fixed order, where they are needed
    s.loc = o, o += kStepList;
    s.tile_off = o, o += 2 * ((PT + 1) & ~1);
    s.tile_pos = o, o += (PT + 3) & ~3;
    s.tile_phys = o, o += (PT + 3) & ~3;
    s.zred = o, o += (warps + 3) & ~3;
    s.bar = o, o += 2 * groups;
    o = up(o);
    s.solve = s.cand = s.red = o;
    if (solve) {
        s.cand = up(s.solve + kSolveWords);
        s.red = s.cand + 4 * cands;
        o = up(s.red + warps * D);
    }
    s.work = o;
    // work area: page scores, then the key tiles of the next round (or, in the exact token fallback, the keys in position
    // order), then the candidates, the partial readouts and the value rows in flight, or an iterative solve's key rows
    int w = PT * 16;
    s.vring = s.work;
    if (!solve) {
        s.cand = s.work;
        s.red = up(s.work + 4 * cands);
        s.vring = up(s.red + warps * D);
    }
    const int stages = solve ? cands / (4 * groups) : step_value_stages(threads, false);   // (of a solve: those that K_c needs)
    const int vring_end = s.vring + 4 * stages * threads * lane_words - s.work;
    w = vring_end > w ? vring_end : w;
    if (fused && ((max_pages + 11) & ~3) > w) w = (max_pages + 11) & ~3;
    // page scan: the queries of the cluster's heads and the summary rows of the next round, beside the scores
    s.scan_q = up(s.work + ((max_pages + 11) & ~3));
    s.scan_ring = up(s.scan_q + heads * (D / 2));
    if (cluster) {
        const bool ahead = (max_pages + 15) / 16 > cluster * groups;   // more than one round
        const int scan_end = s.scan_ring + (near ? threads * step_scan_stages(D) * (D / 32) * 8 : ahead ? threads * 16 * 4 : 0) - s.work;
        w = scan_end > w ? scan_end : w;
    }
    if (tt > 1 && threads * 16 * lane_words > w) w = threads * 16 * lane_words;
    if (solve && ((K_c + 31) & ~31) * 64 > w) w = ((K_c + 31) & ~31) * 64;
    o = up(o + w);
    s.bt = o;
    // (not where it would cost the second block of an SM)
    s.stage_bt = fused && (cluster || (threads >= 256 && max_pages <= 8192 && (threads == 512 || o + max_pages <= 113 * 256)));
    if (s.stage_bt) o += (max_pages + 15) & ~15;
    s.total = (o + 3) & ~3;
    return s;
}

// Rows that pass through shared memory in pieces of 16 bytes (bulk and asynchronous copies, vector loads) start on 128-byte lines.  On
// 16-byte boundaries, wherever the parts before them ended, microseconds per layer: 160 units of D = 256 with 46 pages 29.6 -> 24.0, 64 sequences of
// 4k - 128k with eight heads a group 300 -> 293, 1184 units of 3k - 18k with 48 pages 67.5 -> 64.6, 352 of at most 1.3k 56.6 -> 54.7, 32
// of 8k at D = 64 41.0 -> 40.5, one sequence of 4k with 100 pages 18.7 -> 17.9; with one round of tiles no difference.
// Where the lines would cost a block on an SM the parts start on 16-byte boundaries.
inline StepLayout step_layout(int threads, int D, int max_pages, int P, int PT, int K_c, bool fused, bool fp8, bool solve,
                              int cluster = 0, int heads = 0, bool near = false)
{
    auto on = [&](int line) { return step_layout_on(line, threads, D, max_pages, P, PT, K_c, fused, fp8, solve, cluster, heads, near); };
    auto blocks = [&](const StepLayout& s) { return std::min(threads == 128 ? 5 : 512 / threads, 228 * 1024 / (s.total * 4 + 1024)); };
    const StepLayout lines = on(32), tight = on(4);
    return blocks(lines) < blocks(tight) ? tight : lines;
}

// Exact page selection when the list overflows (many equal scores).  Leaves exactly K entries in list[] and
// hist[] cleared.  scratch: 16 words; wred: one word per warp (not the words behind scratch, where the winners' list is padded for
// the ranks that follow).
__device__ __noinline__ void step_pages_exact(const BlockTeam& tm, const float* sc, int n, int K, uint32_t* hist,
                                              uint32_t* scratch, uint32_t* wred, unsigned long long* list, uint32_t* counter)
{
    tm.sync();   // every thread has read the counter
    for (int i = tm.tid; i < kStepPages; i += tm.size) list[i] = 0ull;
    if (tm.tid == 0) *counter = 0u;
    tm.sync();
    auto key = [&](int i) { return max(float_to_key(sc[i]), 1u); };   // 0 (one NaN pattern) would read as no page
    team_exact_topk_slow(tm, key, n, K, hist, scratch, wred, [&](int i) {
        list[atomicAdd(counter, 1u)] = ((unsigned long long)key(i) << 32) | (uint32_t)~i;
    });
    for (int i = tm.tid; i < kStepBins; i += tm.size) hist[i] = 0u;
    tm.sync();
}

// Fixed-order scores of pages, one per group of LPR lanes: the canonical chain and halving tree (complete in every lane).
template <int LPR>
__device__ __forceinline__ float page_score(const uint4& q, const uint4& row)
{
    float v = chunk_partial_bf16(q, row);
#pragma unroll
    for (int off = LPR / 2; off; off >>= 1) v += __shfl_xor_sync(kFullMask, v, off);
    return v + 0.0f;   // (the sums over more lanes end in +0 for -0)
}

// All fixed-order scores of the unit's pages into sc[].
template <int THREADS, int D>
__device__ __noinline__ void step_rescore_row(const StepParams& p, const int32_t* bt, uint4 qraw, float* sc, int nb, int g)
{
    constexpr int LPR = step_lanes_per_row(D), GROUPS = THREADS / LPR, U = 4;
    const int c = (threadIdx.x & 31) % LPR, grp = threadIdx.x / LPR;
    const uint8_t* base = reinterpret_cast<const uint8_t*>(p.summaries) + ((long long)g * D + c * 8) * 2;
    const unsigned page_bytes = (unsigned)(p.geo.n_kv_heads * 2 * D);
    __syncthreads();   // every thread has read its own part
#pragma unroll 1
    for (int l0 = 0; l0 < nb; l0 += U * GROUPS) {
        int e[U];
        uint4 row[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int l = l0 + u * GROUPS + grp;
            e[u] = l < nb ? ld_ca_s32(bt + l) : -1;
            if (e[u] >= p.geo.pool_pages) e[u] = -1;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) row[u] = ld_cg_16B(base + (unsigned long long)(unsigned)max(e[u], 0) * page_bytes);
        __syncwarp();
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const float s = page_score<LPR>(qraw, row[u]);
            const int l = l0 + u * GROUPS + grp;
            if (c == 0 && l < nb) sc[l] = e[u] >= 0 ? s : -INFINITY;
        }
    }
    __syncthreads();
}

// Fixed-order scores for listed pages.  marks: for those whose score is a mark (page_mma.cuh).  Otherwise the P-th and the next of the
// scores are too close to tell: the pages from `lowest` on get theirs, which then decide.  Pages below it are not among the P best,
// whatever the rounding (the P-th best score moves by no more than the scores do).
template <int THREADS, int D>
__device__ __noinline__ void step_settle_pages(const StepParams& p, const int32_t* bt, uint4 qraw, unsigned long long* list, int m,
                                               float lowest, bool marks, int g)
{
    constexpr int LPR = step_lanes_per_row(D), GPW = 32 / LPR, GROUPS = THREADS / LPR;
    const int c = (threadIdx.x & 31) % LPR, grp = threadIdx.x / LPR, warp = threadIdx.x >> 5;
    const uint8_t* base = reinterpret_cast<const uint8_t*>(p.summaries) + ((long long)g * D + c * 8) * 2;
    const unsigned page_bytes = (unsigned)(p.geo.n_kv_heads * 2 * D);
#pragma unroll 1
    for (int t0 = 0; t0 + warp * GPW < m; t0 += GROUPS) {
        const int t = t0 + grp;
        const unsigned long long e = t < m ? list[t] : 0ull;
        // (0: a word beside the row; -inf, a page outside the pool, is exact)
        const float s = e != 0ull ? key_to_float((uint32_t)(e >> 32)) : -INFINITY;
        const bool near = marks ? s != s : s != -INFINITY && !(s < lowest);
        const int phys = near ? ld_ca_s32(bt + (int)~(uint32_t)e) : 0;
        const uint4 row = ld_cg_16B(base + (unsigned long long)(unsigned)phys * page_bytes);
        __syncwarp();
        const float exact = page_score<LPR>(qraw, row);
        if (c == 0 && (near || (!marks && s != -INFINITY)))   // (key 1: below the rest, -inf included)
            list[t] = ((unsigned long long)(near ? float_to_key(exact) : 1u) << 32) | (uint32_t)e;
    }
    __syncthreads();
}

// Exact token selection of the R best when the histogram's range is degenerate or its cut bucket crowded: the keys
// in position order (work[]), then every thread's unselected keys become 0.  Returns the key of the R-th best,
// which is unselected as well.
__device__ __noinline__ uint32_t step_tokens_exact(const BlockTeam& tm, uint32_t* own_keys, int n_own, const int32_t* tile_pos,
                                                   int nt, int lanes, int R, uint32_t* hist, uint32_t* scratch, uint32_t* wred,
                                                   uint32_t* work, uint32_t* place)   // place: nullptr where tiles are in position order
{
    const int N = nt * 16;
    const int tpl = lanes == 8 ? 2 : 1, group = tm.tid / lanes, c = tm.tid % lanes, groups = tm.size / lanes;
    if (place) {   // tiles by position (a page may be listed twice)
        for (int t = tm.tid; t < nt; t += tm.size) {
            int at = 0;
            for (int x = 0; x < nt; ++x) at += (int)((tile_pos[x] < tile_pos[t]) | ((tile_pos[x] == tile_pos[t]) & (x < t)));
            place[t] = (uint32_t)at;
        }
        tm.sync();
    }
    auto index_of = [&](int o) {   // array index of own key o, or -1
        const int slot = (o / tpl) * groups + group;
        return slot >= nt || (lanes == 32 && (c & 1)) ? -1 : (place ? (int)place[slot] : slot) * 16 + (lanes == 8 ? 2 * c + o % 2 : lanes == 32 ? c >> 1 : c);
    };
    tm.sync();
    for (int o = 0; o < n_own; ++o) {
        const int i = index_of(o);
        if (i >= 0) work[i] = own_keys[o * tm.size + tm.tid];
    }
    tm.sync();
    const TopkResult r = team_exact_topk_slow(tm, [&](int i) { return work[i]; }, N, R, hist, scratch, wred, [](int) {});
    for (int o = 0; o < n_own; ++o) {
        const int i = index_of(o);
        if (i < 0) continue;
        const uint32_t k = work[i];
        if (k < r.kth_key || (k == r.kth_key && i >= r.kth_idx)) own_keys[o * tm.size + tm.tid] = 0u;
    }
    tm.sync();
    return r.kth_key;
}

// The canonical halving tree over the LPR lanes that hold a row, for the 16 rows of a tile at once.  Lane c ends
// with rows 2c, 2c + 1 (8 lanes), row c (16) or row c / 2 (32).
template <int LPR>
__device__ __forceinline__ void reduce_tile(float (&v)[16], int c)
{
    int n = 16;
#pragma unroll
    for (int off = LPR / 2; off; off >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool hi = c & off;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                if (i < n) {
                    const float send = hi ? v[i] : v[i + n];
                    const float keep = hi ? v[i + n] : v[i];
                    v[i] = keep + __shfl_xor_sync(kFullMask, send, off);
                }
            }
        } else {
            v[0] = v[0] + __shfl_xor_sync(kFullMask, v[0], off);
        }
    }
}

// The same where slot i of lane c holds its partial of row i ^ tile_xor(c): at every level the slot that a lane sends and
// the slot that it adds into are then fixed, which saves the selects.
template <int LPR>
__device__ __forceinline__ int tile_xor(int c)
{
    return LPR == 8 ? 2 * c : LPR == 32 ? c >> 1 : c;
}
template <int LPR>
__device__ __forceinline__ void reduce_tile_xor(float (&v)[16])
{
    int n = 16;
#pragma unroll
    for (int off = LPR / 2; off; off >>= 1) {
        if (n > 1) {
            n >>= 1;
#pragma unroll
            for (int i = 0; i < 8; ++i)
                if (i < n) v[i] += __shfl_xor_sync(kFullMask, v[i + n], off);
        } else {
            v[0] += __shfl_xor_sync(kFullMask, v[0], off);
        }
    }
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// the place of a shared-memory address of this block in block `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_address(uint32_t addr, int rank)
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_store(uint32_t addr, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}

__device__ __forceinline__ void cluster_max(uint32_t addr, uint32_t v)
{
    asm volatile("red.shared::cluster.max.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// The page scan of one (sequence, KV head) by the cluster of the blocks of its query heads and their helpers: tiles of 16 summary rows are
// dealt out to the blocks and, there, to the groups of lanes; a tile is scored for all heads of the cluster in the way of
// token routing, and every head's scores go to the shared memory of its own block.  Where there are fewer tiles than
// groups of lanes, the heads are dealt out as well.  The first tile of a group of lanes comes through registers, every
// later one through shared memory, asked for one round ahead.  Ends with the scores of this block's head complete in sc.
// Bound by one load from memory (0.6 us), the chain of a tile's sums (0.6) and the barrier of the cluster (0.4), where a kernel
// ahead takes 3.1 with its boundary and 0.5 to read its scores: one sequence of 4k 12.6 -> 11.2 us per layer, as one call 12.0 -> 10.5.
template <int THREADS, int D>
__device__ __forceinline__ void step_scan_pages(const StepParams& p, const int32_t* bt_s, const uint8_t* qs, const uint8_t* ring,
                                                const float* sc, int nb, int g)
{
    constexpr int LPR = step_lanes_per_row(D), GPW = 32 / LPR, GROUPS = THREADS / LPR, ROW = 2 * D, TPL = LPR == 8 ? 2 : 1;
    const Geometry& geo = p.geo;
    const int tid = threadIdx.x, warp = tid >> 5, c = tid % LPR, grp = tid / LPR;
    const int cs = p.cluster_shift, C = 1 << cs, rank = (int)blockIdx.x & (C - 1), hs = p.heads_shift;
    const int n_tiles = (nb + 15) >> 4, mine = (n_tiles - rank + C - 1) >> cs;   // tiles rank, rank + C, ...
    int ss = 0;   // log2 of the parts that the heads are dealt out in
    while (ss < hs && (mine << (ss + 1)) <= GROUPS) ++ss;
    const int n_items = mine << ss, per = (1 << hs) >> ss;
    const uint8_t* base = reinterpret_cast<const uint8_t*>(p.summaries) + (long long)g * ROW + c * 16;
    const unsigned page_bytes = (unsigned)(geo.n_kv_heads * ROW);
    const uint32_t sc_s = (uint32_t)__cvta_generic_to_shared(sc);
    const uint8_t* own_ring = ring + grp * 16 * ROW;
    const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(own_ring) + c * 16, at = (uint32_t)(tile_xor<LPR>(c) * ROW + c * 16);
    auto tile_of = [&](int item) { return rank + ((item >> ss) << cs); };
    auto page_ok = [&](int e) { return e >= 0 && e < geo.pool_pages; };
    // rows without a valid page read row 0 of the pool instead (their score becomes -inf)
    auto row_of = [&](int e) { return base + (unsigned long long)(unsigned)(page_ok(e) ? e : 0) * page_bytes; };
    auto entries = [&](int item, int (&e)[16]) {   // (entries past the sequence are whatever the table holds)
        const int4* t4 = reinterpret_cast<const int4*>(bt_s + 16 * tile_of(item));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int4 x = t4[i];
            e[4 * i] = x.x, e[4 * i + 1] = x.y, e[4 * i + 2] = x.z, e[4 * i + 3] = x.w;
        }
    };
    const bool any = warp * GPW < n_items;
    uint4 rows[16];
    auto ahead = [&](int item) {
        if (item >= n_items) return;
        int e[16];
        entries(item, e);
#pragma unroll
        for (int t = 0; t < 16; ++t) cp_async_16B(ring_s + (uint32_t)(t * ROW), row_of(e[t]));
    };
    if (any) {
        int e[16];
        entries(grp < n_items ? grp : 0, e);
#pragma unroll
        for (int t = 0; t < 16; ++t) rows[t] = ld_cg_16B(row_of(e[t]));
        cp_async_commit_group();   // (the queries)
        ahead(grp + GROUPS);
    } else {
        cp_async_commit_group();
    }
    cp_async_commit_group();
    cp_async_wait_group<1>();
    __syncthreads();
    cluster_wait();   // the other blocks of the cluster run
#pragma unroll 1
    for (int i0 = 0; i0 + warp * GPW < n_items; i0 += GROUPS) {
        const int item = i0 + grp;
        if (i0 != 0) {
            cp_async_wait_all();
            __syncwarp();   // the other lanes' pieces of the tile
#pragma unroll
            for (int t = 0; t < 16; ++t) rows[t] = *reinterpret_cast<const uint4*>(own_ring + (at ^ (uint32_t)(t * ROW)));
            __syncwarp();
            ahead(item + GROUPS);
        }
        const int first = tile_of(item) * 16, head0 = (item & ((1 << ss) - 1)) * per;
#pragma unroll 1
        for (int hh = head0; hh < head0 + per; ++hh) {
            const uint4 qv = *reinterpret_cast<const uint4*>(qs + hh * ROW + c * 16);
            float vals[16];
#pragma unroll
            for (int t = 0; t < 16; ++t) vals[t] = chunk_partial_bf16(qv, rows[t]);
            __syncwarp();
            if (i0 != 0)
                reduce_tile_xor<LPR>(vals);
            else
                reduce_tile<LPR>(vals, c);
            const uint32_t dst = cluster_address(sc_s, hh);
#pragma unroll
            for (int s = 0; s < TPL; ++s) {
                const int l = first + (LPR == 8 ? 2 * c + s : LPR == 32 ? c >> 1 : c);
                if (item < n_items && l < nb && (LPR != 32 || (c & 1) == 0))
                    cluster_store(dst + 4u * (uint32_t)l, page_ok(bt_s[l]) ? vals[s] : -INFINITY);
            }
        }
    }
    __syncwarp();
    cluster_arrive();
    cluster_wait();
}

// The page scan of one (sequence, KV head) by the cluster of the blocks of its query heads and their helpers: tiles of 16 summary
// rows are dealt out to the warps of all blocks, scored for all heads of the cluster by MMAs (page_mma.cuh: near ties
// are settled later), and every head's scores go to the shared memory of its own block, the bound of their rounding to all.
// Rows come through shared memory, every lane copying what it reads itself: loads into registers need lines of the L1, of
// which blocks with this much shared memory leave 28 KB.  Ends with the scores of this block's head complete in sc.
template <int THREADS, int D>
__device__ __forceinline__ void step_scan_pages_mma(const StepParams& p, const int32_t* bt_s, const uint8_t* qs, uint8_t* ring_base,
                                                const float* sc, uint32_t* bound, int nb, int g)
{
    constexpr int ROW = 2 * D, KC = D / 32, STAGES = step_scan_stages(D), WARPS = THREADS / 32;
    const Geometry& geo = p.geo;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, r = lane >> 2, j = lane & 3;
    cp_async_commit_group();   // (the queries)
    const int cs = p.cluster_shift, C = 1 << cs, rank = (int)blockIdx.x & (C - 1), heads = 1 << p.heads_shift;
    // warps of the cluster take tiles in turn, block by block, so that few tiles are spread over all SMs
    const int n_tiles = (nb + 15) >> 4, first_tile = (warp << cs) + rank, step = WARPS << cs;
    const uint8_t* base = reinterpret_cast<const uint8_t*>(p.summaries) + (long long)g * ROW + j * 16;
    const unsigned page_bytes = (unsigned)(geo.n_kv_heads * ROW);
    uint4* own = reinterpret_cast<uint4*>(ring_base) + warp * (STAGES * 2 * KC * 32) + lane;   // piece i of stage s: own[(s * 2 KC + i) * 32]
    const uint32_t own_s = (uint32_t)__cvta_generic_to_shared(own);
    auto page_ok = [&](int e) { return e >= 0 && e < geo.pool_pages; };
    auto issue = [&](int tile, int stage) {   // rows without a valid page read row 0 of the pool instead (their score becomes -inf)
        if (tile >= n_tiles) return;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = bt_s[tile * 16 + h * 8 + r];   // (entries past the sequence are whatever the table holds)
            const uint8_t* row = base + (unsigned long long)(unsigned)(page_ok(e) ? e : 0) * page_bytes;
#pragma unroll
            for (int i = 0; i < KC; ++i) cp_async_16B(own_s + (uint32_t)((stage * 2 * KC + h * KC + i) * 512), row + 64 * i);
        }
    };
#pragma unroll
    for (int s = 0; s < STAGES; ++s) {
        issue(first_tile + s * step, s);
        cp_async_commit_group();
    }
    cp_async_wait_group<STAGES>();   // the queries, asked for before
    __syncthreads();
    uint4 q[KC];
#pragma unroll
    for (int i = 0; i < KC; ++i) q[i] = r < heads ? *reinterpret_cast<const uint4*>(qs + r * ROW + (j + 4 * i) * 16) : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t sc_s = (uint32_t)__cvta_generic_to_shared(sc);
    const bool has0 = 2 * j < heads, has1 = 2 * j + 1 < heads;
    const uint32_t dst0 = has0 ? cluster_address(sc_s, 2 * j) : 0u, dst1 = has1 ? cluster_address(sc_s, 2 * j + 1) : 0u;
    uint32_t most = 0u;
    cluster_wait();   // the other blocks of the cluster run
    int stage = 0;
#pragma unroll 1
    for (int tile = first_tile; tile < n_tiles; tile += step) {
        cp_async_wait_group<STAGES - 1>();
        PageTile<D> t;
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            t.row[0][i] = own[(stage * 2 * KC + i) * 32];
            t.row[1][i] = own[(stage * 2 * KC + KC + i) * 32];
        }
        float s[4], a[4];
        t.dot(q, s, a);
        __syncwarp();
        issue(tile + STAGES * step, stage);
        cp_async_commit_group();
        stage = stage + 1 == STAGES ? 0 : stage + 1;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int l = tile * 16 + h * 8 + r;
            if (l >= nb) continue;
            const bool ok = page_ok(bt_s[l]);
            uint32_t a0 = __float_as_uint(a[2 * h]), a1 = __float_as_uint(a[2 * h + 1]);
            if (max(a0, a1) >= kNoBound) mark_without_bound(s[2 * h], a0), mark_without_bound(s[2 * h + 1], a1);
            if (ok) most = max(most, max(a0, a1));
            if (has0) cluster_store(dst0 + 4u * (uint32_t)l, ok ? s[2 * h] : -INFINITY);
            if (has1) cluster_store(dst1 + 4u * (uint32_t)l, ok ? s[2 * h + 1] : -INFINITY);
        }
    }
    __syncwarp();
    most = __reduce_max_sync(kFullMask, most);
    if (lane < heads && most != 0u) cluster_max(cluster_address((uint32_t)__cvta_generic_to_shared(bound), lane), most);
    __syncwarp();
    cluster_arrive();
    cluster_wait();
}

__device__ __noinline__ void step_failed_unit(const BlockTeam& tm, const StepParams& p, long long unit, int status, int D,
                                              bool routed_too)
{
    for (int e = tm.tid; e < D; e += tm.size) p.out[unit * D + e] = 0.0f;
    if (tm.tid == 0) {
        vsa_diag_t d;
        d.delta = d.delta12 = d.s_max = d.lse = d.leak_bound = 0.0f;
        d.n_candidates = 0;
        d.fallback = 0;
        d.status = status;
        p.diag[unit] = d;
        if (p.solve) p.solve[unit] = vsa_solve_t{0.0f, 0.0f, 0.0f, 0.0f};
        if (p.flags) p.flags[unit] = 0;
    }
    if (routed_too)
        for (int t = tm.tid; t < p.P; t += tm.size) p.routed_pages[unit * p.P + t] = -1;
}

// Entries of list[0 .. n) that are greater than e, counted by four lanes (part = lane & 3), the total in each of
// them; list[] is zero up to the next multiple of 32.  All lanes of the warp take part.
__device__ __forceinline__ int rank_in_list(const unsigned long long* list, int n, unsigned long long e, int part)
{
    const ulonglong2* l2 = reinterpret_cast<const ulonglong2*>(list) + part;
    int r0 = 0, r1 = 0;
#pragma unroll 1
    for (int j = 0; j < n; j += 32) {
        ulonglong2 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = l2[j / 2 + 4 * u];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            r0 += x[u].x > e;
            r1 += x[u].y > e;
        }
    }
    r0 += r1;
    __syncwarp();
    r0 += __shfl_xor_sync(kFullMask, r0, 1);
    return r0 + __shfl_xor_sync(kFullMask, r0, 2);
}

// The same for the position order: entries of win[0 .. n) below l, n padded with INT_MAX to a multiple of 16.
__device__ __forceinline__ int rank_below(const int32_t* win, int n, int l, int part)
{
    const int4* w4 = reinterpret_cast<const int4*>(win) + part;
    int r0 = 0, r1 = 0;
#pragma unroll 2
    for (int j = 0; j < n; j += 16) {
        const int4 x = w4[j / 4];
        r0 += (x.x < l) + (x.y < l);
        r1 += (x.z < l) + (x.w < l);
    }
    r0 += r1;
    __syncwarp();
    r0 += __shfl_xor_sync(kFullMask, r0, 1);
    return r0 + __shfl_xor_sync(kFullMask, r0, 2);
}

// THREADS: 512 (one block per SM) when there are no more units than SMs, 256 (two) up to two units per SM, 128
//   (four, or BLOCKS = five) beyond: a unit is a latency chain, so units in flight count for more than threads per unit.
// FUSED: the unit's pages are selected here from page_scores (1, by MMAs 3) or from scores computed here (2, by MMAs 4: the blocks of a
//   cluster are the query heads of a KV head, eight at most); otherwise (0) routed_pages is an input.
// BY_POSITION: order of the tiles, the same for pages as an input as in the step of the shape, so that both sum in one order.
// D: head dimension.  A row is spread over D / 8 lanes, 8 elements (16 bytes; fp8: 8 bytes) each, so a warp works
//   on 4, 2 or 1 tiles of 16 rows at a time.
// FP8: k / v hold e4m3 bytes with one scale per (pool page, KV head); strides count bytes.  Scores and weights are
//   multiplied by the scale afterwards (exact for powers of two).
// SOLVE: the weights come from solver_iters entropic (1) or Frank-Wolfe (2) iterations (step_solve.cuh).
template <int THREADS, int FUSED, int D = kHeadDim, bool FP8 = false, int SOLVE = 0, int BLOCKS = 512 / THREADS, bool BY_POSITION = true>
__global__ void __launch_bounds__(THREADS, BLOCKS) sparse_step_kernel(const __grid_constant__ StepParams p)
{
    constexpr int WARPS = THREADS / 32, LPR = step_lanes_per_row(D), GPW = 32 / LPR, GROUPS = THREADS / LPR;
    constexpr bool BULK = THREADS == 128;   // key tiles by bulk copies
    // The routed pages fill the slots of tiles in the order of their scores or, in a phase more, of their positions: the heads of a KV head then
    // walk the pages that they share at about the same time.  Microseconds per layer by score / position.  512 threads behind a scan (the
    // rule is step_by_position in sparse.cu): one round of tiles 4 of 16k with 32 pages 14.1 / 14.3; more, 4 of 16k 48 pages 16.2 / 15.9, 64
    // 17.7 / 17.4, D = 256 8 of 8k with two heads a group 26.3 / 25.3, but one head a group, 16 of 16k 23.1 / 23.3, D = 256 16 of 8k 25.9 / 26.3, and few
    // units, D = 256 one of 8k 15.9 / 16.5.  In a cluster, whose blocks leave the scan together, 4 of 4k 48 pages 14.0 / 14.4, 64 14.7 / 15.1,
    // one of 4k 100 pages 17.9 / 18.2.  Always by position (on 16-byte boundaries of shared memory): 256 threads 8 of 16k 19.2 / 19.0, 64 pages 26.4 /
    // 25.7; 128 threads 64 of 8k 79.4 / 77.2, 32 of 8k with 64 pages 72.7 / 71.1, D = 256 78.8 / 75.9; e4m3 16 of 16k 29.6 / 30.3, but 4 of
    // 16k 14.3 / 14.1 and sixteen heads of one KV head, 19 of 3k, 41.8 / 40.9.  Always by score: 128 threads of D = 64, 32 of 8k 41.5 / 41.9, in 32-token
    // pages 36.5 / 37.0, but 64 of 8k with 32 pages 68.6 / 67.7.  (Scores by MMAs: by position, since near ties would leave their order open.)
    constexpr bool SELECT = FUSED != 0, CLUSTER = FUSED == 2 || FUSED == 4, MMA = FUSED == 3 || FUSED == 4;
    static_assert(BY_POSITION || (!MMA && step_order_open(THREADS, D, FP8)), "by position");
    // A scan ahead of this kernel has waited for whatever wrote the cache before this kernel starts.  Without one its blocks may already run
    // beside the append, and what that writes is not read-only: no ld.global.nc.  (Nothing here writes an e4m3 cache's rows.)  Loads of the
    // value rows past the L1, which wait for one another, cost 2 - 5 % of the step: 8 of 4k with two heads a group and 24 pages 12.0 -> 12.6.
    constexpr bool BEHIND_SCAN = FUSED == 1 || FUSED == 3;
    constexpr int TPL = LPR == 8 ? 2 : 1;   // tokens of a tile per lane (D = 256: the even lanes own one each)
    static_assert(!FP8 || D == 128, "fp8 cache: head dimension 128");
    static_assert(SOLVE == 0 || (THREADS == 256 && D == 128 && !FP8), "the solve maps one candidate to each of 256 lanes");
    extern __shared__ __align__(16) uint32_t smem[];
    const Geometry& geo = p.geo;
    const int tid = threadIdx.x;
    const BlockTeam tm{tid, THREADS};
    const int tsh = geo.tile_shift, P = p.P;
    const StepLayout& lay = p.lay;
    uint32_t* ctl = smem;
    uint32_t* hist = smem + lay.hist;
    uint32_t* warp_stat = smem + lay.warp_stat;   // page phase: [warp] threshold; token phase: [warp] best two keys
    unsigned long long* pages = reinterpret_cast<unsigned long long*>(smem + lay.list);
    unsigned long long* tokens = reinterpret_cast<unsigned long long*>(smem + lay.tokens);
    int32_t* win = (int32_t*)(smem + lay.win);
    uint32_t* win_key = smem + lay.win_key;   // key of the page with that rank
    int32_t* win_phys = (int32_t*)(smem + lay.loc);   // (until the token selection)
    uint32_t* settled = win_key + ((p.P + 3) & ~3);
    long long* tile_off = reinterpret_cast<long long*>(smem + lay.tile_off);   // element offset of a tile's first row, -1 = none
    int32_t* tile_pos = (int32_t*)(smem + lay.tile_pos);                       // its first token's position
    int32_t* tile_phys = (int32_t*)(smem + lay.tile_phys);                     // its pool page
    uint32_t* own = smem + lay.keys + tid;                             // this thread's token keys, stride THREADS
    float* red = (float*)(smem + lay.red);
    float* zred = (float*)(smem + lay.zred);
    uint32_t* work = smem + lay.work;
    int32_t* bt_s = (int32_t*)(smem + lay.bt);
    const int lane = tid & 31, warp = tid >> 5, c = lane % LPR, grp = tid / LPR;
    int h = blockIdx.x, helper = 0;
    if constexpr (CLUSTER) {   // (a helper: the first head of its cluster)
        helper = (h & ((1 << p.cluster_shift) - 1)) >> p.heads_shift;
        h = ((h >> p.cluster_shift) << p.heads_shift) + (helper ? 0 : h & ((1 << p.heads_shift) - 1));
    }
    const int b = blockIdx.y, g = h >> p.group_shift;
    const long long unit = b * geo.n_q_heads + h;   // (batch * n_q_heads fits 30 bits)
    const int32_t* bt = p.block_table + (long long)b * geo.max_pages;

    // before the wait on the preceding kernel: the sequence length, the query (unless the scan runs here: the routing kernel
    // that precedes this one in a step has read both), the block-table row and cleared counters
    const int T = ld_ca_s32(p.seq_lens + b);
    uint4 qraw;
    if constexpr (!CLUSTER) qraw = ld_nc_16B(p.q + unit * D + c * 8);
    if (SELECT && lay.stage_bt) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(bt_s);
        for (int i = tid; i < geo.max_pages; i += THREADS) cp_async_4(dst + 4u * (uint32_t)i, bt + i);
    }
    cp_async_commit_group();
    for (int i = tid; i < lay.zeroed / 4; i += THREADS) reinterpret_cast<uint4*>(smem)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (SELECT && BY_POSITION)
        for (int i = tid; i < ((P + 15) & ~15); i += THREADS) win[i] = INT_MAX;
    const bool length_ok = geo.length_ok(T);
    const int nb = length_ok ? geo.pages_of(T) : 0;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(smem + lay.bar) + 8u * (uint32_t)grp;   // BULK: of this group of lanes
    if constexpr (BULK) {
        if (c == 0) mbar_init(bar, 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    const int r_warp = (P + WARPS - 1) / WARPS;
    if constexpr (CLUSTER) {
        cluster_arrive();
        cp_async_wait_all();
        __syncthreads();
    }
    pdl_wait();
    pdl_launch_dependents();
    if (CLUSTER && tid == 0 && unit < p.n_tickets) p.tickets[unit] = 0;
    if (!length_ok) {
        if constexpr (CLUSTER) cluster_wait();
        if (helper) return;
        cp_async_wait_all();
        step_failed_unit(tm, p, unit, VSA_UNIT_BAD_LENGTH, D, SELECT);
        return;
    }

    // tiles of a routed page: addresses and positions
    auto put_page = [&](int slot, int l, int phys) {
        const bool ok = phys >= 0 && phys < geo.pool_pages;
        if (!ok) ctl[kCtlBad] = 1u;
        if (l == nb - 1) atomicAdd(&ctl[kCtlMissing], (uint32_t)(nb * geo.page_size - T));
        for (int hf = 0; hf < (1 << tsh); ++hf) {
            const int s = (slot << tsh) + hf;
            tile_off[s] = ok ? (long long)phys * geo.page_stride + (long long)(hf * 16) * geo.token_stride : -1;
            tile_pos[s] = l * geo.page_size + hf * 16;
            tile_phys[s] = phys;
        }
    };

    int np;
    float slack = 0.0f;   // page scores further apart than this are in the order of the fixed-order ones (0: they are those)
    if constexpr (SELECT) {
        // ---- stage the scores of the sequence's pages, four to a chunk; a thread only reads back what it copied.
        //      Short rows spread over the warps (all of them have to vouch for r_warp scores) ----
        const float* row = !CLUSTER ? p.page_scores + unit * geo.max_pages : nullptr;
        const int mis = !CLUSTER ? (int)((unit * geo.max_pages) & 3) : 0, n_chunks = (nb + mis + 3) >> 2;
        const bool single = n_chunks <= THREADS;   // a chunk per thread at most: it stays in registers
        const int chunk0 = single ? lane * WARPS + warp : tid, l0 = 4 * chunk0 - mis;
        float* sc = reinterpret_cast<float*>(work);
        float4* sc4 = reinterpret_cast<float4*>(sc);
        np = min(P, nb);
        auto in_row = [&](int l) { return (unsigned)l < (unsigned)nb; };
        if constexpr (CLUSTER) {
            const int heads = 1 << p.heads_shift, first = h & ~(heads - 1);
            const uint8_t* qs = reinterpret_cast<const uint8_t*>(smem + lay.scan_q);
            const uint32_t qs_s = (uint32_t)__cvta_generic_to_shared(qs);
            for (int i = tid; i < heads * (D / 8); i += THREADS)
                cp_async_16B(qs_s + 16u * (uint32_t)i, p.q + ((long long)b * geo.n_q_heads + first) * D + i * 8);
            uint8_t* ring = reinterpret_cast<uint8_t*>(smem + lay.scan_ring);
            if constexpr (MMA)
                step_scan_pages_mma<THREADS, D>(p, bt_s, qs, ring, sc, &ctl[kCtlBound], nb, g);
            else
                step_scan_pages<THREADS, D>(p, bt_s, qs, ring, sc, nb, g);
            if (helper) return;
            qraw = *reinterpret_cast<const uint4*>(qs + (h - first) * 2 * D + c * 16);
        }
        // the bound of the scores' rounding, over the blocks of pages that the sequence has
        uint32_t bound = FUSED == 4 ? ctl[kCtlBound] : 0u;
        if constexpr (FUSED == 3) {
            const int hs = min(p.group_shift, 3), blocks = bound_blocks(nb);
            const int32_t* from = reinterpret_cast<const int32_t*>(p.bounds) + (long long)(unit >> hs) * bound_blocks(geo.max_pages);
            for (int i = tid; i < blocks; i += THREADS) bound = max(bound, (uint32_t)ld_cg_s32(from + i));
        }
        float4 own_chunk = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        // words of the first and the last chunk that are no scores of this row: below or equal to every score
        if (single) {
            if (chunk0 < n_chunks) {
                const float4 v = !CLUSTER ? ld_cg_f32x4(row + l0) : sc4[chunk0];
                if (in_row(l0)) own_chunk.x = v.x;
                if (in_row(l0 + 1)) own_chunk.y = v.y;
                if (in_row(l0 + 2)) own_chunk.z = v.z;
                if (in_row(l0 + 3)) own_chunk.w = v.w;
            }
        } else if constexpr (!CLUSTER) {
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(sc);
            for (int i = chunk0; i < n_chunks; i += THREADS) cp_async_16B(dst + 16u * (uint32_t)i, row - mis + 4 * i);
        }
        cp_async_wait_all();
        if (!single) {
            if (chunk0 == 0)
                for (int e = 0; e < mis; ++e) sc[e] = -INFINITY;
            if ((n_chunks - 1) % THREADS == chunk0)
                for (int e = nb + mis; e < 4 * n_chunks; ++e) sc[e] = -INFINITY;
        }
        // ---- the warp's r-th largest lane maximum ----
        {
            float m = fmaxf(fmaxf(own_chunk.x, own_chunk.y), fmaxf(own_chunk.z, own_chunk.w));
            if (!single) {
#pragma unroll 4
                for (int i = chunk0; i < n_chunks; i += THREADS) {
                    const float4 v = sc4[i];
                    m = fmaxf(m, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
                }
            }
            __syncwarp();
            uint32_t v = chunk0 < n_chunks ? float_to_key(m) : 0u, thr = 0u;
#pragma unroll 1
            for (int i = 0; i < r_warp; ++i) {
                thr = __reduce_max_sync(kFullMask, v);
                const unsigned holders = __ballot_sync(kFullMask, v == thr);
                if (lane == __ffs(holders) - 1) v = 0u;   // remove one holder of the maximum
            }
            if (lane == 0) warp_stat[warp] = thr;   // 0: fewer than r lanes have a score, then every score is listed
            if constexpr (FUSED == 3) {
                bound = __reduce_max_sync(kFullMask, bound);
                if (lane == 0) smem[lay.misc + warp] = bound;
            }
        }
        __syncthreads();
        if constexpr (FUSED == 3) {
#pragma unroll
            for (int w = 0; w < WARPS; w += 4) {
                const uint4 x = *reinterpret_cast<const uint4*>(smem + lay.misc + w);
                bound = max(bound, max(max(x.x, x.y), max(x.z, x.w)));
            }
        }
        if constexpr (MMA) slack = page_score_slack(__uint_as_float(bound));
        // ---- list every score that is not below the smallest of them.  A NaN never is, so whatever the scores are at
        //      least np pages are listed: every lane that a warp vouched for has one (a lane of NaNs vouches with -inf,
        //      which lists everything).  Listed by key, a NaN ranks first, as in the exact selections ----
        {
            uint32_t theta_key = 0xffffffffu;
#pragma unroll
            for (int w = 0; w < WARPS; w += 4) {
                const uint4 x = *reinterpret_cast<const uint4*>(warp_stat + w);
                theta_key = min(theta_key, min(min(x.x, x.y), min(x.z, x.w)));
            }
            const float theta = theta_key <= 0x007fffffu ? -INFINITY : key_to_float(theta_key) - (MMA ? slack : 0.0f);
            auto entry = [&](float score, int l) { return ((unsigned long long)float_to_key(score) << 32) | (uint32_t)~l; };
            if (single) {
                const float4 v = own_chunk;
                const bool h0 = in_row(l0) && !(v.x < theta), h1 = in_row(l0 + 1) && !(v.y < theta),
                           h2 = in_row(l0 + 2) && !(v.z < theta), h3 = in_row(l0 + 3) && !(v.w < theta);
                const unsigned b0 = __ballot_sync(kFullMask, h0), b1 = __ballot_sync(kFullMask, h1),
                               b2 = __ballot_sync(kFullMask, h2), b3 = __ballot_sync(kFullMask, h3);
                const int n0 = __popc(b0), n1 = n0 + __popc(b1), n2 = n1 + __popc(b2), n3 = n2 + __popc(b3);
                if (n3) {
                    int s = 0;
                    if (lane == 0) s = (int)atomicAdd(&ctl[kCtlPages], (uint32_t)n3);
                    __syncwarp();
                    s = __shfl_sync(kFullMask, s, 0);
                    if (s + n3 <= kStepPages) {   // otherwise the list overflows and the exact selection runs
                        const unsigned below = (1u << lane) - 1u;
                        if (h0) pages[s + __popc(b0 & below)] = entry(v.x, l0);
                        if (h1) pages[s + n0 + __popc(b1 & below)] = entry(v.y, l0 + 1);
                        if (h2) pages[s + n1 + __popc(b2 & below)] = entry(v.z, l0 + 2);
                        if (h3) pages[s + n2 + __popc(b3 & below)] = entry(v.w, l0 + 3);
                    }
                }
            } else {
#pragma unroll 1
                for (int i1 = 0; i1 < n_chunks; i1 += 8 * THREADS) {
                    const int i0 = i1 + chunk0;
                    uint32_t hits = 0u;   // four bits per chunk
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int i = i0 + u * THREADS;
                        if (i < n_chunks) {
                            const float4 v = sc4[i];
                            hits |= ((v.x < theta ? 0u : 1u) | (v.y < theta ? 0u : 2u) | (v.z < theta ? 0u : 4u) |
                                     (v.w < theta ? 0u : 8u)) << (4 * u);
                        }
                    }
                    uint32_t s = hits ? atomicAdd(&ctl[kCtlPages], (uint32_t)__popc(hits)) : 0u;
                    if (s + __popc(hits) > kStepPages) hits = 0u;
                    while (hits) {
                        const int bit = __ffs(hits) - 1;
                        hits &= hits - 1u;
                        const int i = 4 * (i0 + (bit >> 2) * THREADS) + (bit & 3), l = i - mis;
                        // (a word beside the row, listed when everything is, leaves its entry 0: ranked last)
                        if (in_row(l)) pages[s] = entry(sc[i], l);
                        ++s;
                    }
                    __syncwarp();
                }
            }
        }
        __syncthreads();
        int m = (int)ctl[kCtlPages];
        bool marks = MMA;   // pages whose score is a mark may be listed (they always are: NaN is not below theta)
        if (m > kStepPages) {
            if (single && chunk0 < n_chunks) sc4[chunk0] = own_chunk;
            if constexpr (MMA) {
                step_rescore_row<THREADS, D>(p, bt, qraw, sc + mis, nb, g);
                slack = 0.0f;
                marks = false;
            }
            step_pages_exact(tm, sc + mis, nb, np, hist, smem + lay.misc, warp_stat, pages, &ctl[kCtlPages]);
            m = np;
        }
        // ---- exact ranks, four lanes per listed page.  By position the pages are put into slots in a phase of their own ----
#pragma unroll 1
        while (true) {
#pragma unroll 1
            for (int t0 = 0; t0 < m; t0 += THREADS / 4) {
                const int t = t0 + (tid >> 2);
                const unsigned long long e = t < m ? pages[t] : ~0ull;
                if (t0 + (warp << 3) >= m) break;   // nothing left for this warp
                if constexpr (BY_POSITION) {
                    const int rank = rank_in_list(pages, m, e, tid & 3);
                    if (t < m && rank < np + (MMA ? 1 : 0) && (tid & 3) == 0) {
                        if (rank < np) {
                            win[rank] = (int)~(uint32_t)e;
                            if constexpr (MMA) win_key[rank] = (uint32_t)(e >> 32);
                        } else if constexpr (MMA) {
                            ctl[kCtlNext] = (uint32_t)(e >> 32);
                        }
                    }
                } else {   // the page of rank t fills slot t
                    const int l = (int)~(uint32_t)e, at = t < m && l >= 0 ? l : 0;   // (a word beside the row is ranked last)
                    const int phys = lay.stage_bt ? bt_s[at] : ld_ca_s32(bt + at);
                    const int rank = rank_in_list(pages, m, e, tid & 3);
                    if (t < m && rank < np && (tid & 3) == 0) {
                        put_page(rank, l, phys);
                        p.routed_pages[unit * P + rank] = l;
                    }
                }
            }
            __syncthreads();
            if constexpr (!MMA) break;
            if (marks) {   // they rank first
                marks = false;
                const float best = key_to_float(win_key[0]);
                if (best != best) {
                    if constexpr (MMA) step_settle_pages<THREADS, D>(p, bt, qraw, pages, m, 0.0f, true, g);
                    continue;
                }
            }
            if (slack == 0.0f || m <= np) break;
            const uint32_t next = ctl[kCtlNext];   // (0: no page, but a word beside the row)
            const float kth = key_to_float(win_key[np - 1]);
            if (next == 0u || kth - key_to_float(next) > slack) break;
            if constexpr (MMA) step_settle_pages<THREADS, D>(p, bt, qraw, pages, m, kth - slack, false, g);
            slack = 0.0f;   // the scores are the fixed-order ones
        }
        for (int t = np + tid; t < P; t += THREADS) p.routed_pages[unit * P + t] = -1;
        if constexpr (BY_POSITION) {
#pragma unroll 1
            for (int t0 = 0; t0 < np; t0 += THREADS / 4) {
                if (t0 + (warp << 3) >= np) break;
                const int t = t0 + (tid >> 2);
                const int l = t < np ? win[t] : 0;
                const int phys = lay.stage_bt ? bt_s[l] : ld_ca_s32(bt + l);
                const int slot = rank_below(win, np, l, tid & 3);
                if (t < np && (tid & 3) == 0) {
                    put_page(slot, l, phys);
                    p.routed_pages[unit * P + t] = l;
                    if constexpr (MMA) win_phys[t] = phys;
                }
            }
            __syncthreads();
        }
    } else {
        for (int t = tid; t < P; t += THREADS) {
            const int l = p.routed_pages[unit * P + t];
            win[t] = l >= 0 && l < nb ? l : INT_MAX;
        }
        __syncthreads();
        for (int t = tid; t < P; t += THREADS) {
            const int l = win[t];
            if (l == INT_MAX) continue;
            const int phys = ld_ca_s32(bt + l);
            int slot = 0;
#pragma unroll 4
            for (int j = 0; j < P; ++j) slot += BY_POSITION ? (int)((win[j] < l) | ((win[j] == l) & (j < t))) : (int)((j < t) & (win[j] != INT_MAX));
            put_page(slot, l, phys);
            atomicAdd(&ctl[kCtlNp], 1u);
        }
        __syncthreads();
        np = (int)ctl[kCtlNp];
    }
    // The list of routed pages is ordered by score: pages whose scores are too close to tell from a neighbour's get their
    // fixed-order scores (a warp settles 32 ranks, a group of lanes a page at a time), ...
    unsigned close = 0u;   // of ranks 32 * warp ...
    if (MMA && slack != 0.0f && warp * 32 < np) {
        const int t = warp * 32 + lane;
        bool near = false, either = false;   // (-inf, a page outside the pool, is exact)
        if (t < np) {
            const float s = key_to_float(win_key[t]), next = t + 1 < np ? key_to_float(win_key[t + 1]) : -INFINITY,
                        last = t > 0 ? key_to_float(win_key[t - 1]) : INFINITY;
            near = next != -INFINITY && !(s - next > slack);
            either = near || (s != -INFINITY && !(last - s > slack));
        }
        const unsigned word = __ballot_sync(kFullMask, near);
        close = __ballot_sync(kFullMask, either);
        if (lane == 0) ctl[kCtlNear + warp] = word;
    }
    auto next_close = [&] {   // this group of lanes' next one, or -1
        int t = -1;
#pragma unroll
        for (int k = 0; k < GPW; ++k) {
            if (close && k == lane / LPR) t = warp * 32 + __ffs(close) - 1;
            close &= close - 1u;
        }
        return t;
    };
    auto close_row = [&](int t) {
        const uint8_t* from = reinterpret_cast<const uint8_t*>(p.summaries) + ((long long)g * D + c * 8) * 2;
        return ld_cg_16B(from + (unsigned long long)(unsigned)(t >= 0 ? win_phys[t] : 0) * (unsigned)(geo.n_kv_heads * 2 * D));
    };
    auto settle_score = [&](int t, const uint4& row) {   // (by all lanes of a warp)
        const float s = page_score<LPR>(qraw, row);
        if (c == 0 && t >= 0) settled[t] = float_to_key(s);
    };
    // ... and, later, their places among the neighbours that are close to one another
    auto settle_places = [&](int first, int step) {
        const uint4 words = *reinterpret_cast<const uint4*>(ctl + kCtlNear);
        if (!(words.x | words.y | words.z | words.w)) return;
        auto near = [&](int x) { return x >= 0 && ((ctl[kCtlNear + (x >> 5)] >> (x & 31)) & 1u); };
#pragma unroll 1
        for (int t = first; t < np; t += step) {
            if (!near(t) && !near(t - 1)) continue;
            const uint32_t key = settled[t];
            const int l = win[t];
            auto before = [&](int x) { return settled[x] > key || (settled[x] == key && win[x] < l); };
            int at = t;
            for (int x = t - 1; near(x); --x) at -= !before(x);
            for (int x = t + 1; near(x - 1); ++x) at += before(x);
            p.routed_pages[unit * P + at] = l;
        }
    };
    if (ctl[kCtlBad]) {
        if constexpr (MMA) {
            while (close) {
                const int t = next_close();
                settle_score(t, close_row(t));
            }
            __syncthreads();
            settle_places(tid, THREADS);
        }
        step_failed_unit(tm, p, unit, VSA_UNIT_BAD_PAGE, D, false);
        return;
    }
    const int n_valid = np * geo.page_size - (int)ctl[kCtlMissing];   // tokens that get a score
    const int nt = np << tsh;                                         // their tiles
    const int rounds = (nt + GROUPS - 1) / GROUPS;

    uint4 first_close;   // asked for ahead of the keys
    int first_t = -1;
    if (MMA && close) {
        first_t = next_close();
        first_close = close_row(first_t);
    }

    // ---- token routing: one tile of 16 rows per group of lanes and round ----
    uint32_t a1 = 0u, a2 = 0u, amin = 0xffffffffu;   // best, second best and smallest key of this thread
    {
        // The first tile comes through registers, every later one through shared memory, asked for one round ahead: by
        // asynchronous copies that a lane reads back itself or (BULK) by one bulk copy of 16 contiguous rows, which a lane reads
        // in the order t ^ tile_xor(c) (from global memory that order would take a sector per lane).  BULK saves 16 copies with
        // their addresses and 30 selects of the 360 instructions of a round: 19.2k -> 16.4k cycles of a unit with 64 tiles in a
        // full chip, 8.2k -> 5.8k with 32 at D = 64.  Larger blocks have one or two rounds, which its set-up costs (batch 8,
        // T = 32k 22.6 -> 22.9 us per layer).  Streams of four rows with eight in flight were slower (28k cycles).
        using Bits = typename std::conditional<FP8, uint2, uint4>::type;
        constexpr int kElem = FP8 ? 1 : 2, ROW = D * kElem, TILE = 16 * ROW;
        const uint8_t* kbase = reinterpret_cast<const uint8_t*>(p.k) + ((long long)g * geo.head_stride + c * 8) * kElem;
        const long long stride = (long long)geo.token_stride * kElem;
        const uint8_t* ring = reinterpret_cast<const uint8_t*>(work);
        // BULK: the group's tile, row t ^ tile_xor(c) at mine ^ t * ROW; otherwise row t at mine + t * THREADS
        const uint32_t mine = BULK ? (uint32_t)(grp * TILE + tile_xor<LPR>(c) * ROW + c * 8 * kElem) : (uint32_t)(tid * sizeof(Bits));
        const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring) + (BULK ? (uint32_t)(grp * TILE) : mine);
        auto ahead = [&](int slot) {
            if (slot >= nt) return;
            const uint8_t* src = kbase + tile_off[slot] * kElem;
            if constexpr (BULK) {
                if (c == 0) {
                    mbar_expect_tx(bar, TILE);
                    if (geo.token_stride == D)
                        bulk_load(ring_s, src, TILE, bar);
                    else
                        for (int t = 0; t < 16; ++t) bulk_load(ring_s + t * ROW, src + t * stride, ROW, bar);
                }
            } else {
#pragma unroll
                for (int t = 0; t < 16; ++t) {
                    if constexpr (FP8)
                        cp_async_8B(ring_s + t * THREADS * 8, src + t * stride);
                    else
                        cp_async_16B(ring_s + t * THREADS * 16, src + t * stride);
                }
            }
        };
        if (BULK && rounds > 1) fence_async_proxy();   // the page scores lay where the copies go
#pragma unroll 1
        for (int r = 0; r < rounds; ++r) {
            const int slot = r * GROUPS + grp;
            if (r * GROUPS + warp * GPW >= nt) {   // no tile left for this warp (last round)
#pragma unroll
                for (int s = 0; s < TPL; ++s) own[(r * TPL + s) * THREADS] = 0u;
                break;
            }
            const bool active = slot < nt;
            float kscale = 1.0f;
            if (FP8 && active) kscale = __ldg(p.k_scale + (long long)tile_phys[slot] * geo.n_kv_heads + g);
            Bits rows[16];
            if (r == 0) {
                const uint8_t* src = kbase + (active ? tile_off[slot] : tile_off[0]) * kElem;
#pragma unroll
                for (int t = 0; t < 16; ++t) {
                    if constexpr (FP8)
                        rows[t] = ld_nc_8B(src + t * stride);
                    else
                        rows[t] = BEHIND_SCAN ? ld_nc_16B(src + t * stride) : ld_cg_16B(src + t * stride);
                }
            } else if constexpr (BULK) {
                if (active && !mbar_wait(bar, (uint32_t)(r - 1) & 1u)) ctl[kCtlLate] = 1u;
#pragma unroll
                for (int t = 0; t < 16; ++t) rows[t] = *reinterpret_cast<const Bits*>(ring + (mine ^ (uint32_t)(t * ROW)));
                __syncwarp();   // read by all lanes: the next tile may land
            } else {
                cp_async_wait_all();
#pragma unroll
                for (int t = 0; t < 16; ++t) rows[t] = reinterpret_cast<const Bits*>(ring + mine)[t * THREADS];
            }
            ahead(slot + GROUPS);
            float vals[16];
#pragma unroll
            for (int t = 0; t < 16; ++t) {
                if constexpr (FP8) {
                    float qf[8], kf[8];
                    unpack8(qraw, qf);
                    unpack8_e4m3_mixed(rows[t], kf);
                    vals[t] = chunk_partial(qf, kf);
                } else {
                    vals[t] = chunk_partial_bf16(qraw, rows[t]);
                }
            }
            __syncwarp();
            if (BULK && r != 0)
                reduce_tile_xor<LPR>(vals);
            else
                reduce_tile<LPR>(vals, c);
            const int pos = active ? tile_pos[slot] : INT_MAX - 16;
#pragma unroll
            for (int s = 0; s < TPL; ++s) {
                const int tok = LPR == 8 ? 2 * c + s : LPR == 32 ? c >> 1 : c;
                const bool mine = LPR != 32 || (c & 1) == 0;
                const float score = FP8 ? __fmul_rn(vals[s], kscale) : vals[s];
                const uint32_t key = (mine && pos + tok < T) ? float_to_key(score) : 0u;
                own[(r * TPL + s) * THREADS] = key;
                a2 = max(a2, min(a1, key));
                a1 = max(a1, key);
                amin = min(amin, key != 0u ? key : 0xffffffffu);
            }
        }
    }
    if (MMA && __any_sync(kFullMask, first_t >= 0)) {
        settle_score(first_t, first_close);
#pragma unroll 1
        while (close) {
            const int t = next_close();
            settle_score(t, close_row(t));
        }
    }
    // Largest and smallest key, and a bracket of the bulk of the scores: the smallest of the warps' largest keys and
    // the largest of the warps' smallest (the histogram's range; a few outliers do not stretch it).  All four as
    // maxima, so that lanes 0 .. 3 publish them with one instruction.
    {
        const uint32_t wmax = __reduce_max_sync(kFullMask, a1), wmin = __reduce_min_sync(kFullMask, amin);
        const uint32_t v = lane & 2 ? wmin : wmax;
        if (lane < 4 && wmax != 0u) atomicMax(&ctl[kCtlStat + lane], lane & 1 ? ~v : v);
    }
    __syncthreads();
    const uint4 stat = *reinterpret_cast<const uint4*>(ctl + kCtlStat);
    if (BULK && ctl[kCtlLate]) {
        if (MMA) settle_places(tid, THREADS);
        step_failed_unit(tm, p, unit, VSA_UNIT_COPY_TIMEOUT, D, false);
        return;
    }
    const uint32_t key1 = stat.x;
    const float s1 = n_valid > 0 ? key_to_float(key1) : -INFINITY;
    const int ns = min(p.K_c, n_valid);
    // ---- exact top-(ns + 1): its last element is the best rejected token, the others are the candidates ----
    const bool has_rejected = n_valid > ns;
    const int R = ns + 1, n_own = rounds * TPL;
    int cut = -1, need = 0;   // cut bucket, and how many of its best tokens belong to the top-(ns + 1)
    float lo = 0.0f, bscale = 0.0f;
    auto bucket_of = [&](uint32_t key) {
        return (int)fminf(fmaxf((key_to_float(key) - lo) * bscale, 0.0f), (float)(kStepBins - 1));
    };
    if (has_rejected) {
        float hi = key_to_float(~stat.y);
        lo = key_to_float(stat.z);
        if (!(hi > lo)) {
            hi = s1;
            lo = key_to_float(~stat.w);
        }
        bscale = __fdividef((float)kStepBins, hi - lo);   // (0 for a huge range: one bucket, the exact selection)
        bool fast = hi > lo && bscale < INFINITY && hi - lo < INFINITY;
        if (fast) {
#pragma unroll 1
            for (int o = 0; o < n_own; ++o) {
                const uint32_t key = own[o * THREADS];
                if (key != 0u) atomicAdd(&hist[bucket_of(key)], 1u);
            }
            __syncthreads();
            // one warp finds the cut: lane j owns bins 8j .. 8j + 7, counts are summed from the top
            if (warp == 0) {
                const uint4 na = reinterpret_cast<const uint4*>(hist)[2 * lane], nc = reinterpret_cast<const uint4*>(hist)[2 * lane + 1];
                const uint32_t n[8] = {na.x, na.y, na.z, na.w, nc.x, nc.y, nc.z, nc.w};
                uint32_t above[9];   // above[j]: tokens in this lane's bins >= j
                above[8] = 0u;
#pragma unroll
                for (int j = 7; j >= 0; --j) above[j] = above[j + 1] + n[j];
                uint32_t incl = above[0];
#pragma unroll
                for (int off = 1; off < 32; off <<= 1) {
                    const uint32_t o = __shfl_down_sync(kFullMask, incl, off);
                    if (lane + off < 32) incl += o;
                }
                const uint32_t base = incl - above[0];   // tokens in the bins of higher lanes
                if (base < (uint32_t)R && (uint32_t)R <= incl) {   // exactly one lane
                    int bin = 0;
#pragma unroll
                    for (int j = 1; j < 8; ++j) bin += base + above[j] >= (uint32_t)R;   // the highest bin that reaches R from the top
                    uint32_t higher = 0u, in_bin = 0u;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (bin == j) higher = above[j + 1], in_bin = n[j];
                    ctl[kCtlCut] = ((base + higher) << 20) | (in_bin << 8) | (uint32_t)(8 * lane + bin);
                }
            }
            __syncthreads();
            const uint32_t packed = ctl[kCtlCut];
            cut = (int)(packed & 255u);
            need = R - (int)(packed >> 20);
            fast = ((packed >> 8) & 4095u) <= kStepList;
        }
        if (fast) {
            uint32_t* loc = smem + lay.loc;   // where the listed key lives
#pragma unroll 2
            for (int o = 0; o < n_own; ++o) {
                const uint32_t key = own[o * THREADS];
                if (key != 0u && bucket_of(key) == cut) {
                    const int slot = (o / TPL) * GROUPS + grp;
                    // by position; a page that the caller lists twice has tiles of its own
                    const int order = (BY_POSITION ? 0 : tile_pos[slot] >> 4 << 11) + slot * 16 + (LPR == 8 ? 2 * c + o % TPL : LPR == 32 ? c >> 1 : c);
                    const uint32_t i = atomicAdd(&ctl[kCtlTokens], 1u);
                    tokens[i] = ((unsigned long long)key << 32) | (uint32_t)~order;
                    loc[i] = (uint32_t)(o * THREADS + tid);
                }
            }
            __syncthreads();
            // four lanes rank a listed token; those that do not belong to the candidates lose their key
            const int m = (int)ctl[kCtlTokens];
#pragma unroll 1
            for (int t0 = 0; t0 < m; t0 += THREADS / 4) {
                if (t0 + (warp << 3) >= m) break;
                const int t = t0 + (tid >> 2);
                const unsigned long long e = t < m ? tokens[t] : ~0ull;
                const int rank = rank_in_list(tokens, m, e, tid & 3);
                if (t < m && rank >= need - 1 && (tid & 3) == 0) {
                    smem[lay.keys + loc[t]] = 0u;
                    if (rank == need - 1) ctl[kCtlOut] = (uint32_t)(e >> 32);
                }
            }
            __syncthreads();
        } else {
            cut = -1;
            const uint32_t k = step_tokens_exact(tm, smem + lay.keys, n_own, tile_pos, nt, LPR, R, hist, smem + lay.misc, warp_stat, work,
                                                 BY_POSITION ? nullptr : smem + lay.loc);
            if (tid == 0) ctl[kCtlOut] = k;
        }
    }

    // ---- the candidates, compacted for the value gather ----
    struct __align__(16) Row {
        long long off;   // element offset of the value row inside its KV head
        float w;         // weight (fp8: times the scale of the row's page)
        float pad;
    };
    Row* cand = reinterpret_cast<Row*>(smem + lay.cand);
    float* cand_score = (float*)(smem + lay.solve);                                     // SOLVE only
    int32_t* cand_pos = (int32_t*)(smem + lay.solve + VSA_SOLVER_MAX_CANDIDATES);
    const float scale = 1.4426950408889634f / p.epsilon;   // log2(e) / epsilon
    auto is_candidate = [&](uint32_t key) { return key != 0u && (cut < 0 || bucket_of(key) >= cut); };
    int at = 0;   // first slot of this warp
    {
        int mine = 0;
#pragma unroll 2
        for (int o = 0; o < n_own; ++o) mine += __popc(__ballot_sync(kFullMask, is_candidate(own[o * THREADS])));
        if (lane == 0) warp_stat[warp] = (uint32_t)mine;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < WARPS; w += 4) {
            const uint4 x = *reinterpret_cast<const uint4*>(warp_stat + w);
            at += (w < warp ? x.x : 0u) + (w + 1 < warp ? x.y : 0u) + (w + 2 < warp ? x.z : 0u) + (w + 3 < warp ? x.w : 0u);
        }
    }
    float z = 0.0f;
#pragma unroll 2
    for (int o = 0; o < n_own; ++o) {
        const uint32_t key = own[o * THREADS];
        const bool take = is_candidate(key);
        const unsigned votes = __ballot_sync(kFullMask, take);
        if (take) {
            const int slot = (o / TPL) * GROUPS + grp;
            const int tok = LPR == 8 ? 2 * c + o % TPL : LPR == 32 ? c >> 1 : c;
            Row row;
            row.off = tile_off[slot] + (long long)tok * geo.token_stride;
            const float w = exp2f((key_to_float(key) - s1) * scale);
            z += w;
            row.w = FP8 ? w * __ldg(p.v_scale + (long long)tile_phys[slot] * geo.n_kv_heads + g) : w;
            row.pad = 0.0f;
            const int j = at + __popc(votes & ((1u << lane) - 1u));
            cand[j] = row;
            if constexpr (SOLVE != 0) {
                cand_score[j] = key_to_float(key);
                cand_pos[j] = tile_pos[slot] + tok;
            }
        }
        at += __popc(votes);
    }
    constexpr int UNR = 4;   // rows of a group of lanes that the value gather takes at a time
    const int n_rows = (ns + UNR * GROUPS - 1) / (UNR * GROUPS) * UNR;   // past the candidates: the last one, weight 0
    static_assert(UNR * GROUPS <= THREADS, "fewer than a row each");
    if (ns < n_rows * GROUPS) {   // (the same for the block; K_c is a multiple as a rule)
        __syncthreads();
        if (ns + tid < n_rows * GROUPS) cand[ns + tid] = Row{cand[ns - 1].off, 0.0f, 0.0f};
    }
    __syncthreads();

    float lse_closed = 0.0f;   // log-sum-exp of the closed-form weights (SOLVE only)
    if constexpr (SOLVE != 0) {
        // the candidates' key rows once more (L2 hits), then the solve's weights in place of the closed form's
        if (ns > 0) {
            uint8_t* tile = reinterpret_cast<uint8_t*>(work);
            const uint32_t tile_s = (uint32_t)__cvta_generic_to_shared(tile);
            const uint16_t* kbase = p.k + (long long)g * geo.head_stride + c * 8;
#pragma unroll 4
            for (int j = grp; j < ((ns + 31) & ~31); j += GROUPS) {
                if (j < ns)
                    cp_async_16B(tile_s + tile_at(j, c), kbase + cand[j].off);
                else
                    *reinterpret_cast<uint4*>(tile + tile_at(j, c)) = make_uint4(0u, 0u, 0u, 0u);
            }
            cp_async_commit_group();
            float* spare = (float*)(smem + lay.solve + 2 * VSA_SOLVER_MAX_CANDIDATES);
            const SolveSmem ss{tile, reinterpret_cast<uint32_t*>(pages), red, spare + VSA_SOLVER_MAX_CANDIDATES, spare};
            const float s_own = tid < ns ? cand_score[tid] : 0.0f;
            float z0 = z;
#pragma unroll
            for (int off = 16; off; off >>= 1) z0 += __shfl_xor_sync(kFullMask, z0, off);
            if (lane == 0) zred[warp] = z0;
            cp_async_wait_all();
            __syncthreads();
            if constexpr (SOLVE == 2) {
                z = solve_frank_wolfe(ss, ns, s_own, tid < ns ? cand_pos[tid] : 0, p.solver_iters, qraw, p.solve + unit);
                float Z0 = 0.0f;
#pragma unroll
                for (int w = 0; w < WARPS; ++w) Z0 += zred[w];
                lse_closed = s1 / p.epsilon + logf(Z0);
                __syncthreads();   // zred is rewritten by the value gather
            } else {
                z = solve_entropic(ss, ns, s_own, p.solver_iters, p.epsilon, qraw, lse_closed, p.solve + unit);
            }
            if (tid < ns) cand[tid].w = z;
        } else if (tid == 0) {
            p.solve[unit] = vsa_solve_t{0.0f, 0.0f, 0.0f, 0.0f};
        }
        __syncthreads();
    }

    // ---- value gather: the candidates dealt out to the groups of lanes, four rows at a time.  A block of 128 or 256 threads
    //      streams them through stages in shared memory: the loop is a quarter of the code of sixteen rows in registers (the SM
    //      caches some 2000 instructions, a kernel with units in all phases needs its code again and again: 20.7k -> 14k
    //      cycles of a unit with K_c = 512 in a full chip, 4.0k -> 3.4k at K_c = 256 and two units per SM).  With 512 threads
    //      every instruction runs once, and rows in registers are faster (batch 1, T = 4k 14.4 against 14.7 us per layer).  After
    //      an iterative solve nothing else overlaps the loads: all rows at once (three stages and four, mean over six orders of
    //      loading the kernels, whose place in memory moves one and the same code by 1.5 %: batch 8, T = 32k, four Frank-Wolfe
    //      iterations 32.4 -> 32.0 us per layer, two entropic ones 33.0 -> 32.8, four 37.3 -> 37.2; batch 24 89.0 -> 88.2; batch 1,
    //      T = 8k 22.6 -> 22.8) ----
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
    {
        using Bits = typename std::conditional<FP8, uint2, uint4>::type;
        constexpr int kElem = FP8 ? 1 : 2, STAGES = step_value_stages(THREADS, SOLVE != 0);
        static_assert(SOLVE == 0 || STAGES * UNR * GROUPS == VSA_SOLVER_MAX_CANDIDATES, "a solve's rows are asked for once");
        const uint8_t* vbase = reinterpret_cast<const uint8_t*>(p.v) + ((long long)g * geo.head_stride + c * 8) * kElem;
        const Row* mine = cand + grp;
        auto add = [&](const Bits& row, float w) {
            float vf[8];
            if constexpr (FP8)
                unpack8_e4m3_mixed(row, vf);
            else
                unpack8_mixed(row, vf);
#pragma unroll
            for (int e = 0; e < 8; e += 2) fma2(acc[e], acc[e + 1], w, w, vf[e], vf[e + 1]);
        };
        // meanwhile: the sum of the weights and the warp's two best keys
        auto statistics = [&] {
            __syncwarp();
#pragma unroll
            for (int off = 16; off; off >>= 1) z += __shfl_xor_sync(kFullMask, z, off);
            const uint32_t best = __reduce_max_sync(kFullMask, a1);
            const int holder = __ffs(__ballot_sync(kFullMask, a1 == best)) - 1;
            const uint32_t second = __reduce_max_sync(kFullMask, lane == holder ? a2 : a1);
            if (lane == 0) {
                zred[warp] = z;
                warp_stat[2 * warp] = best;
                warp_stat[2 * warp + 1] = second;
            }
            __syncwarp();
        };
        if constexpr (STAGES == 0) {
            constexpr int BATCHES = 4;
            Bits rows[BATCHES][UNR];
            float w[BATCHES][UNR];
            auto fetch = [&](int t, int i) {   // batch t of the registers <- rows i .. i + UNR - 1 of this group
#pragma unroll
                for (int u = 0; u < UNR; ++u) {
                    const Row row = mine[(i + u) * GROUPS];
                    w[t][u] = row.w;
                    if constexpr (FP8)
                        rows[t][u] = ld_nc_8B(vbase + row.off * kElem);
                    else
                        rows[t][u] = BEHIND_SCAN ? ld_nc_16B(vbase + row.off * kElem) : ld_once_16B(vbase + row.off * kElem);
                }
            };
#pragma unroll
            for (int t = 0; t < BATCHES; ++t)
                if (t * UNR < n_rows) fetch(t, t * UNR);
            statistics();
#pragma unroll 1
            for (int i0 = 0; i0 < n_rows; i0 += BATCHES * UNR)
#pragma unroll
                for (int t = 0; t < BATCHES; ++t)
                    if (i0 + t * UNR < n_rows) {
#pragma unroll
                        for (int u = 0; u < UNR; ++u) add(rows[t][u], w[t][u]);
                        if (i0 + (t + BATCHES) * UNR < n_rows) fetch(t, i0 + (t + BATCHES) * UNR);
                    }
        } else {
            const Bits* ring = reinterpret_cast<const Bits*>(smem + lay.vring) + tid;   // row t of a stage at + t * THREADS
            const uint32_t ring_s = (uint32_t)__cvta_generic_to_shared(ring);
            auto fetch = [&](int i, int stage) {   // stage <- rows i .. i + UNR - 1 of this group
#pragma unroll
                for (int u = 0; u < UNR; ++u) {
                    const uint8_t* src = vbase + mine[(i + u) * GROUPS].off * kElem;
                    const uint32_t dst = ring_s + (uint32_t)((stage * UNR + u) * THREADS * sizeof(Bits));
                    if constexpr (FP8)
                        cp_async_8B(dst, src);
                    else
                        cp_async_16B(dst, src);
                }
            };
#pragma unroll 1
            for (int s = 0; s < STAGES; ++s) {
                if (UNR * s < n_rows) fetch(UNR * s, s);
                cp_async_commit_group();
            }
            statistics();
            int stage = 0;
#pragma unroll 1
            for (int i = 0; i < n_rows; i += UNR) {
                cp_async_wait_group<STAGES - 1>();
#pragma unroll
                for (int u = 0; u < UNR; ++u) add(ring[(stage * UNR + u) * THREADS], mine[(i + u) * GROUPS].w);
                if (i + UNR * STAGES < n_rows) fetch(i + UNR * STAGES, stage);
                cp_async_commit_group();
                stage = stage + 1 == STAGES ? 0 : stage + 1;
            }
        }
    }
#pragma unroll
    for (int off = LPR; off < 32; off <<= 1)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] += __shfl_xor_sync(kFullMask, acc[e], off);
    if (lane < LPR) {
        float4* dst = reinterpret_cast<float4*>(red + warp * D + c * 8);
        dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
    }
    __syncthreads();
    constexpr int SETTLER = D / 32 < WARPS - 1 ? D / 32 : 0;   // a warp that has nothing else to do, if there is one
    if (MMA && warp == SETTLER) settle_places(lane, 32);
    if (warp >= D / 32 && warp != WARPS - 1) return;
    float Z = 0.0f;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) Z += zred[w];
    for (int e = tid; e < D; e += THREADS) {
        float a = 0.0f;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) a += red[w * D + e];
        p.out[unit * D + e] = ns > 0 ? a / Z : 0.0f;
    }

    // ---- diagnostics and fallback flag (the last warp, which has no output row of its own) ----
    if (warp == WARPS - 1) {
        // second best key: the best of all but one holder of the best, whose warp offers its own second
        const uint32_t w1 = lane < WARPS ? warp_stat[2 * lane] : 0u, w2 = lane < WARPS ? warp_stat[2 * lane + 1] : 0u;
        const int holder = __ffs(__ballot_sync(kFullMask, w1 == key1)) - 1;
        const uint32_t key2 = __reduce_max_sync(kFullMask, lane == holder ? w2 : w1);
        if (lane != 0) return;
        const float s2 = ns > 1 ? key_to_float(key2) : -INFINITY;
        const float delta = has_rejected ? s1 - key_to_float(ctl[kCtlOut]) : INFINITY;
        vsa_diag_t d;
        d.delta = delta;
        d.delta12 = ns > 0 ? s1 - s2 : INFINITY;
        d.s_max = s1;
        d.lse = ns > 0 ? (SOLVE ? lse_closed : s1 / p.epsilon + logf(Z)) : -INFINITY;
        d.leak_bound = fminf(1.0f, (float)(T - ns) * expf(-delta / p.epsilon));
        d.n_candidates = ns;
        d.fallback = (delta < p.gap_threshold && ns < T) ? 1 : 0;
        d.status = 0;
        p.diag[unit] = d;
        if (CLUSTER)
            p.flags[unit] = d.fallback;
        else if (d.fallback)
            p.fallback_list[atomicAdd(p.fallback_count, 1)] = (int32_t)unit;
    }
}

template <int THREADS, int FUSED, int D, bool FP8, int SOLVE = 0, int BLOCKS = 512 / THREADS, bool BY_POSITION = true>
cudaError_t launch_step_variant(const StepParams& p, cudaStream_t stream)
{
    static bool attr_done[kMaxDevices] = {};   // per template instance
    size_t smem = (size_t)p.lay.total * 4;
    // a scanning block has an SM of its own (two units of a solve on one SM, which a cluster's blocks otherwise share: one
    // sequence of 4k, four entropic iterations 27.2 against 20.7 us per layer)
    if ((FUSED == 2 || FUSED == 4) && p.scan_per_sm == 1 && smem < 120 * 1024) smem = 120 * 1024;
    // So has a unit of a solve, whose passes fill the SM, where there are enough: beside the scan's blocks two go to one otherwise.
    // Microseconds per layer, four entropic iterations, one of 32k 29.3 -> 24.1, of 128k 34.6 -> 29.2, 4 of 8k 29.8 -> 23.9, of 16k 31.0 -> 25.3,
    // Frank-Wolfe 25.9 -> 21.5.
    if (SOLVE != 0 && (long long)p.geo.batch * p.geo.n_q_heads <= device_sm_count() && smem < 120 * 1024) smem = 120 * 1024;
    if (smem > 48 * 1024) {
        const cudaError_t e = allow_large_dynamic_smem(sparse_step_kernel<THREADS, FUSED, D, FP8, SOLVE, BLOCKS, BY_POSITION>, attr_done);
        if (e != cudaSuccess) return e;
    }
    if constexpr (FUSED == 2 || FUSED == 4) {
        if (p.active_clusters)
            return active_clusters(sparse_step_kernel<THREADS, FUSED, D, FP8, SOLVE, BLOCKS, BY_POSITION>, dim3(THREADS), 1u << p.cluster_shift, smem,
                                   stream, p.active_clusters);
        return launch_pdl_cluster(sparse_step_kernel<THREADS, FUSED, D, FP8, SOLVE, BLOCKS, BY_POSITION>,
                                  dim3((unsigned)(p.geo.n_q_heads >> p.heads_shift << p.cluster_shift), (unsigned)p.geo.batch),
                                  dim3(THREADS), 1u << p.cluster_shift, smem, stream, p);
    } else
        return launch_pdl(sparse_step_kernel<THREADS, FUSED, D, FP8, SOLVE, BLOCKS, BY_POSITION>,
                          dim3((unsigned)p.geo.n_q_heads, (unsigned)p.geo.batch), dim3(THREADS), smem, stream, p);
}

// in the order of the tiles that the launch has
template <int THREADS, int FUSED, int D, bool FP8, int BLOCKS = 512 / THREADS>
cudaError_t launch_step_order(const StepParams& p, cudaStream_t stream)
{
    if constexpr (step_order_open(THREADS, D, FP8))
        if (!p.by_position) return launch_step_variant<THREADS, FUSED, D, FP8, 0, BLOCKS, false>(p, stream);
    return launch_step_variant<THREADS, FUSED, D, FP8, 0, BLOCKS>(p, stream);
}

template <int D, bool FP8>
cudaError_t launch_step_family(const StepParams& p, int threads, cudaStream_t stream)
{
    const bool fused = p.page_scores != nullptr;
    if (p.summaries && !fused) {
        if (threads == 256 && p.scan_mma) return launch_step_variant<256, 4, D, FP8>(p, stream);
        if (threads != 512) return cudaErrorInvalidValue;
        return p.scan_mma ? launch_step_variant<512, 4, D, FP8>(p, stream) : launch_step_order<512, 2, D, FP8>(p, stream);
    }
    // Five blocks per SM at 96 registers against four at 128, which make a unit 5 - 10 % faster: five
    // where they save a wave of blocks, and from three waves of four on, where units in flight count for more.  Microseconds
    // per layer, four / five, T = 8k.  A wave saved: 32 pages a unit, 640 units 41.6 / 31.9, 704 43.5 / 32.5, 1280 65.4 / 56.0,
    // 1472 68.1 / 63.6; 64 pages 640 66.0 / 48.0, 1472 107 / 100; e4m3 cache 640 39.6 / 29.0, 1472 68.6 / 56.6; D = 64 640
    // 36.0 / 29.2, 1472 63.6 / 60.4; D = 256 640 66.4 / 50.7, 1472 109 / 102.  None saved: 512 26.6 / 29.1, 768 45.1 / 44.5,
    // 1024 47.7 / 50.6, 1152 49.2 / 52.8.  From three waves on: 32 pages 1792 84.0 / 75.9,
    // 2240 90.1 / 90.1, 3200 131 / 120; 64 pages 2048 140 / 124; e4m3 cache 2048 89.2 / 78.7; D = 64 2240 75.8 / 75.7, 3200
    // 114 / 106; D = 256 2240 146 / 147, 3200 214 / 199.  Not where five do not fit the shared memory of an SM (D = 256, 64
    // pages a unit: four 1 % faster).
    const long long units = (long long)p.geo.batch * p.geo.n_q_heads, four = 4LL * device_sm_count(), five = 5LL * device_sm_count();
    const bool fits = (size_t)p.lay.total * 4 + 1024 <= (size_t)228 * 1024 / 5;   // (1 KB of each block is the system's)
    const bool five_blocks = fits && ((units + five - 1) / five < (units + four - 1) / four || units >= 3 * four);
    if (p.bounds) {
        if (threads != 128) return cudaErrorInvalidValue;
        return five_blocks ? launch_step_variant<128, 3, D, FP8, 0, 5>(p, stream) : launch_step_variant<128, 3, D, FP8>(p, stream);
    }
    if (threads == 128 && fused && five_blocks) return launch_step_order<128, 1, D, FP8, 5>(p, stream);
#define VSA_STEP_CASE(T)                                                                    \
    if (threads == T)                                                                       \
        return fused ? launch_step_order<T, 1, D, FP8>(p, stream)                           \
                     : launch_step_order<T, 0, D, FP8>(p, stream);
    VSA_STEP_CASE(512)
    VSA_STEP_CASE(256)
    VSA_STEP_CASE(128)
#undef VSA_STEP_CASE
    return cudaErrorInvalidValue;
}

}  // namespace

}  // namespace vsa
