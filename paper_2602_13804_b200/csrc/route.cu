// Page routing (paper Sec. 7 step 1): score one summary row per page against every query head that
// reads its KV head, then keep the P best pages per query head.
//
//   route_scan_kernel    streams the summary rows (the only part of the step whose traffic grows
//                        with the context length) and writes all page scores to scratch.
//   route_list_kernel    the same where the grid is several waves: the pages that exist, shared evenly.
//   route_select_kernel  one block per (sequence, query head): exact top-P selection.
#include <math.h>

#include <algorithm>

#include "vsa_device.cuh"
#include "vsa_launch.h"
#include "vsa_select.cuh"

namespace vsa {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanWarps = kScanThreads / 32;
constexpr int kBlockPages = 32;      // pages per block-table block (one coalesced 128-byte load per warp)
// Blocks of 32 pages one warp takes at most.  Fewer pay a warp's start-up more often, more leave fewer, longer warps
// and a longer tail.  Microseconds per layer with 2 / 4 / 8 / 16: batch 16, T = 128k 85.4 / 83.4 / 85.3 / 86.8; 64
// sequences of 32k 145 / 141 / 144 / 152; 32 sequences of 16k - 64k 84.4 / 82.9 / 80.9 / 96.1; 64 sequences of
// 4k - 128k at head dimension 64 143 / 132 / 130 / 136.
constexpr int kMaxBlocksPerWarp = 4;
// Table width from which, and sequences up to which, the list scan takes batches of even lengths.
constexpr int kListPages = 2048;
constexpr int kListBatch = 256;

template <int G, int D = kHeadDim>
struct ScanCfg {
    static constexpr int kRowBytes = 2 * D;               // one summary row
    static constexpr int ROWS = G == 1 ? 8 : 16 / G;      // rows per half-warp per round
    static constexpr int VALS = ROWS * G;                 // (row, head) partials per lane per round (8 or 16)
    static constexpr int ROUND_PAGES = 2 * ROWS;          // pages (rows of one KV head) per warp per round
    // ring slots per warp: a power of two (cheap slot index), about 8 KB of rows
    static constexpr int STAGES = 8192 / (ROUND_PAGES * kRowBytes) < 2 ? 2 : 8192 / (ROUND_PAGES * kRowBytes);
    static_assert((STAGES & (STAGES - 1)) == 0, "slot index is R & (STAGES - 1)");
    static constexpr int RING_BYTES = STAGES * ROUND_PAGES * kRowBytes;
    static constexpr int TAB_BYTES = kMaxBlocksPerWarp * kBlockPages * 4;
    static constexpr int RAD_BYTES = STAGES * ROUND_PAGES * 4;   // page radii of the rounds in flight (CERT)
    static constexpr int WARP_BYTES = RING_BYTES + TAB_BYTES + RAD_BYTES;
};

__device__ __forceinline__ void cp_async_16(uint32_t smem_addr, const void* gptr)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr), "l"(gptr) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Warp w of the grid row of sequence b handles KV head (w % n_kv) and the 32-page blocks
// [slice * blocks_per_warp, (slice + 1) * blocks_per_warp), slice = w / n_kv, so the warps of a
// thread block read the summaries of all KV heads of the same pages (2 KB contiguous per page).
// Every lane streams its own 16-byte column of the rows through a private ring in shared memory
// with cp.async (several rounds in flight, no registers held by loads in flight, and no
// cross-thread synchronisation: a lane only ever reads back what it copied itself).  A half-warp
// covers one 256-byte row per copy instruction; the G query heads of the row's group share each
// unpacked element; 16 (row, head) partials are reduced at once.  For G >= 2 lane c takes the
// rows and the heads of a round in the order (r ^ c / G, h ^ c % G), which is what lets the
// reduction run without per-lane selects (reduce_scatter16_xor).
// CERT: the radius of every page (radii[page][kv head], see radii_kernel) is copied into logical page
// order, rad_logical[b][kv head][page], for the certificate that the fused kernel computes.
// D: head dimension (see sparse_kernel.cuh for how a row of 64 or 256 elements maps to the half-warp's lanes).
// PACKED: the rows stay packed and the dot products are mixed-precision FMAs (a shorter chain); otherwise a row is unpacked
// once for the heads of the group (fewer FMA-pipe slots).
template <int G, bool CERT, int D, bool PACKED>
__global__ void __launch_bounds__(kScanThreads, 2)
route_scan_kernel(Geometry geo, const uint16_t* __restrict__ q, const uint16_t* __restrict__ summaries,
                  const int32_t* __restrict__ block_table, const int32_t* __restrict__ seq_lens,
                  float* __restrict__ scores, int blocks_per_warp, int32_t* zero_word, int32_t* zero_words,
                  int zero_count, const float* __restrict__ radii, float* __restrict__ rad_logical)
{
    using Cfg = ScanCfg<G, D>;
    constexpr int ROWS = Cfg::ROWS, VALS = Cfg::VALS, ROUND_PAGES = Cfg::ROUND_PAGES, STAGES = Cfg::STAGES;
    constexpr int kRowBytes = Cfg::kRowBytes, PIECES = D == 256 ? 2 : 1;
    static_assert(D == 128 || ((D == 64 || D == 256) && !CERT), "certificate: head dimension 128 only");
    constexpr bool XOR_MAP = VALS == 16;
    // block-table blocks fetched before the sequence length is known: the warp's whole range
    constexpr int kFirstBlocks = kMaxBlocksPerWarp;
    extern __shared__ __align__(16) uint8_t scan_smem[];
    const int b = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane & 15, gi = lane >> 4;
    const int w = blockIdx.x * (blockDim.x >> 5) + warp;
    const int g = w % geo.n_kv_heads;
    const int slice = w / geo.n_kv_heads;
    const int first_page = slice * blocks_per_warp * kBlockPages;
    const bool has_range = first_page < geo.max_pages;
    const int kr = XOR_MAP ? c / G : 0, kh = XOR_MAP ? c % G : 0;

    // The sequence length and the block-table entries of the first blocks of this warp's range are
    // fetched before the wait on the preceding kernel (they are scheduler state, not the product of a
    // kernel that signals early completion) so that their latency overlaps that kernel's tail.
    // Every index below max_pages is inside the table's row, whatever the sequence length is.
    const int32_t* bt = block_table + (long long)b * geo.max_pages + first_page;
    const int span = min(blocks_per_warp * kBlockPages, geo.max_pages - first_page);
    int T = 0;
    int first_entries[kFirstBlocks];
    if (has_range) {
        T = ld_ca_s32(seq_lens + b);
#pragma unroll
        for (int k = 0; k < kFirstBlocks; ++k) {
            const int i = k * kBlockPages + lane;
            first_entries[k] = i >= span ? -1 : geo.super_pages ? b * geo.max_pages + first_page + i : ld_ca_s32(bt + i);
        }
    }

    pdl_wait();                 // the score scratch may still be read by the previous step's kernels
    pdl_launch_dependents();

    // housekeeping for the kernels that follow in a step: clear the fallback counter and the
    // per-group tickets of the dense pass
    if (blockIdx.y == 0) {
        if (zero_word && blockIdx.x == 0 && threadIdx.x == 0) *zero_word = 0;
        if (zero_words)
            for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < zero_count; i += gridDim.x * blockDim.x)
                zero_words[i] = 0;
    }
    if (!has_range) return;

    const bool lane_has = D != 64 || c < 8;   // this lane holds a piece of every row
    uint4 qraw[G][PIECES];
#pragma unroll
    for (int hh = 0; hh < G; ++hh)
#pragma unroll
        for (int pc = 0; pc < PIECES; ++pc)
            qraw[hh][pc] = lane_has ? ld_nc_16B(q + ((long long)b * geo.n_q_heads + g * G + (hh ^ kh)) * D + pc * 128 + c * 8)
                                    : make_uint4(0u, 0u, 0u, 0u);

    if (geo.super_pages) {
        // the length in super-pages, expressed as a token count so that the page arithmetic below applies
        const int ns = (geo.pages_of(T) + geo.super_pages - 1) / geo.super_pages;
        T = (T > 0 && ns <= geo.max_pages) ? ns * geo.page_size : 0;
    }
    if (!geo.length_ok(T)) return;
    const int nb = geo.pages_of(T);
    if (first_page >= nb) return;
    const int n_pages = min(blocks_per_warp * kBlockPages, nb - first_page);
    const int n_blocks = (n_pages + kBlockPages - 1) / kBlockPages;
    const int n_rounds = (n_pages + ROUND_PAGES - 1) / ROUND_PAGES;

    uint8_t* my_smem = scan_smem + warp * Cfg::WARP_BYTES;
    // [n_blocks * 32] offset of the page's summary row in 16-byte units, -1 = no valid page
    int32_t* off_tab = (int32_t*)(my_smem + Cfg::RING_BYTES);
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(my_smem);
    const int page_units = geo.kv_heads_stored * (kRowBytes / 16);
    auto encode = [&](int p, int i) { return (i < n_pages && p >= 0 && p < geo.pool_pages) ? p * page_units : -1; };
#pragma unroll
    for (int k = 0; k < kFirstBlocks; ++k)
        if (k < n_blocks) off_tab[k * kBlockPages + lane] = encode(first_entries[k], k * kBlockPages + lane);
    float qf[PACKED ? 1 : G][PIECES][8];
    if constexpr (!PACKED)
#pragma unroll
        for (int hh = 0; hh < G; ++hh)
#pragma unroll
            for (int pc = 0; pc < PIECES; ++pc) unpack8(qraw[hh][pc], qf[hh][pc]);
    __syncwarp();

    const int g_stored = g / geo.kv_div;   // the KV head whose summaries this (possibly virtual) head reads
    const uint8_t* srow = reinterpret_cast<const uint8_t*>(summaries) + (long long)g_stored * kRowBytes + c * 16;
    const uint32_t lane_off = (uint32_t)(gi * ROWS * kRowBytes + c * 16);
    int tab_row[ROWS];   // the table entry of this lane's r-th row of a round
#pragma unroll
    for (int r = 0; r < ROWS; ++r) tab_row[r] = gi * ROWS + (r ^ kr);
    // after the reduction this lane owns (row own_r, head own_h) of its half-warp's ROWS rows
    const int own_r = VALS == 16 ? c / G : (c & 7) / G, own_h = c % G;
    const bool owns = VALS == 16 || c < 8;
    float* out_lane = scores + ((long long)b * geo.n_q_heads + g * G + own_h) * geo.max_pages + first_page +
                      gi * ROWS + own_r;
    // CERT: the lane that owns (row, head 0) also moves the row's radius
    const bool rad_lane = CERT && owns && own_h == 0;
    float* rad_ring = (float*)(my_smem + Cfg::RING_BYTES + Cfg::TAB_BYTES);
    const uint32_t rad_ring_s = (uint32_t)__cvta_generic_to_shared(rad_ring);
    float* rad_out = nullptr;
    if constexpr (CERT)
        rad_out = rad_logical + ((long long)b * geo.kv_heads_stored + g / geo.kv_div) * geo.max_pages + first_page +
                  gi * ROWS + own_r;

    // rows without a valid page read row 0 of the pool instead (their result is never stored)
    auto issue = [&](int R) {
        const uint32_t dst = ring + (uint32_t)((R & (STAGES - 1)) * ROUND_PAGES * kRowBytes) + lane_off;
        const int* tab = off_tab + R * ROUND_PAGES;
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            const uint8_t* from = srow + (long long)max(tab[tab_row[r]], 0) * 16;
#pragma unroll
            for (int pc = 0; pc < PIECES; ++pc)
                if (lane_has) cp_async_16(dst + r * kRowBytes + pc * 256, from + pc * 256);
        }
        if constexpr (CERT) {
            if (rad_lane) {
                // off / 16 = page * n_kv_heads: the row of this page in radii[][n_kv_heads]
                const int off = max(tab[gi * ROWS + own_r], 0);
                cp_async_4(rad_ring_s + 4u * (uint32_t)((R & (STAGES - 1)) * ROUND_PAGES + gi * ROWS + own_r),
                           radii + (off >> 4) + g / geo.kv_div);
            }
        }
    };

#pragma unroll
    for (int s = 0; s < STAGES - 1; ++s) {
        if (s < n_rounds) issue(s);
        cp_async_commit();
    }
    for (int R = 0; R < n_rounds; ++R) {
        if (R + STAGES - 1 < n_rounds) issue(R + STAGES - 1);
        cp_async_commit();
        cp_async_wait<STAGES - 1>();   // this lane's copies of round R have landed
        const uint8_t* src = my_smem + (R & (STAGES - 1)) * ROUND_PAGES * kRowBytes + lane_off;
        float vals[16];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
#pragma unroll
            for (int pc = 0; pc < PIECES; ++pc) {
                const uint4 v = lane_has ? *reinterpret_cast<const uint4*>(src + r * kRowBytes + pc * 256)
                                         : make_uint4(0u, 0u, 0u, 0u);
                float kf[8];
                if constexpr (!PACKED) unpack8(v, kf);
#pragma unroll
                for (int hh = 0; hh < G; ++hh) {
                    float part;
                    if constexpr (PACKED)
                        part = chunk_partial_bf16(qraw[hh][pc], v);
                    else
                        part = chunk_partial(qf[hh][pc], kf);
                    vals[r * G + hh] = pc == 0 ? part : vals[r * G + hh] + part;
                }
            }
        }
        float s;
        if constexpr (XOR_MAP) {
            s = reduce_scatter16_xor(vals);
        } else {
#pragma unroll
            for (int i = VALS; i < 16; ++i) vals[i] = 0.0f;
            s = reduce_scatter16(vals, c);
        }
        const int pl = R * ROUND_PAGES + gi * ROWS + own_r;
        if (owns && pl < n_pages) out_lane[R * ROUND_PAGES] = off_tab[pl] >= 0 ? s : -INFINITY;
        if constexpr (CERT) {
            if (rad_lane && pl < n_pages)
                rad_out[R * ROUND_PAGES] =
                    off_tab[pl] >= 0 ? rad_ring[(R & (STAGES - 1)) * ROUND_PAGES + gi * ROWS + own_r] : 0.0f;
        }
    }
}

// ---- the scan over a list of pages, for several waves of blocks ----
// The grid of the kernel above is sized for the longest sequence; in a ragged batch most of its blocks find no page,
// and in any the others run in waves that each pay the start-up of a block.  Here the pages of all sequences, in units of 8,
// form one list that one wave of warps shares evenly: warp w takes KV head w % n_kv and the (w / n_kv)-th range of the
// list, part by part as it crosses sequences.  The start is a longer chain (lengths, their sums, then the table), so
// small batches keep the kernel above (batch 8, T = 32k: 2.4 us less).  DEPTH rounds of a warp's rows are in flight in
// registers.
// Equal shares end together only if the blocks start together, two on every SM.  The kernel is therefore launched in
// stream order, not as a programmatic dependent: scheduled early, its blocks pile up on the SMs that an idle dense block
// of the step before does not hold, and the rest runs as a second wave (64 sequences of 4k - 128k, four heads a group:
// 198 us per layer early, 149 in order, 162 with the kernel above).
constexpr int kUnitPages = 8;
constexpr int kHalfPages = 128;   // pages of one half of a warp's offset table

template <int G>
struct ListCfg {
    static constexpr int ROWS = ScanCfg<G>::ROWS;
    static constexpr int DEPTH = 16 / ROWS > 4 ? 4 : 16 / ROWS;
    static constexpr int WARP_BYTES = 2 * kHalfPages * 4;
};

template <int G>
__global__ void __launch_bounds__(kScanThreads, 2)
route_list_kernel(Geometry geo, const uint16_t* __restrict__ q, const uint16_t* __restrict__ summaries,
                  const int32_t* __restrict__ block_table, const int32_t* __restrict__ seq_lens,
                  float* __restrict__ scores, int ranges, int32_t* zero_word, int32_t* zero_words, int zero_count)
{
    constexpr int ROWS = ScanCfg<G>::ROWS, VALS = ScanCfg<G>::VALS, ROUND_PAGES = ScanCfg<G>::ROUND_PAGES;
    constexpr int DEPTH = ListCfg<G>::DEPTH, RPH = kHalfPages / ROUND_PAGES;   // rounds per half of the table
    constexpr bool XOR_MAP = VALS == 16;
    extern __shared__ __align__(16) uint8_t scan_smem[];
    // [batch + 1] first unit of every sequence, after the offset tables
    int32_t* first_unit = (int32_t*)(scan_smem + kScanWarps * ListCfg<G>::WARP_BYTES);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane & 15, gi = lane >> 4;
    const int w = blockIdx.x * kScanWarps + warp, g = w % geo.n_kv_heads, range = w / geo.n_kv_heads;
    const int kr = XOR_MAP ? c / G : 0, kh = XOR_MAP ? c % G : 0;
    auto pages_in = [&](int b) {   // 0 for an invalid length
        const int T = ld_ca_s32(seq_lens + b);
        return geo.length_ok(T) ? geo.pages_of(T) : 0;
    };
    if (warp == 0) {
        int base = 0;
        for (int b0 = 0; b0 < geo.batch; b0 += 32) {
            const int u = b0 + lane < geo.batch ? (pages_in(b0 + lane) + kUnitPages - 1) / kUnitPages : 0;
            int incl = u;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(kFullMask, incl, off);
                if (lane >= off) incl += o;
            }
            if (b0 + lane < geo.batch) first_unit[b0 + lane] = base + incl - u;
            base += __shfl_sync(kFullMask, incl, 31);
        }
        if (lane == 0) first_unit[geo.batch] = base;
    }
    __syncthreads();
    const int n_units = first_unit[geo.batch];
    int lo = range < ranges ? (int)((long long)n_units * range / ranges) : n_units;
    const int hi = range < ranges ? (int)((long long)n_units * (range + 1) / ranges) : n_units;
    // the sequence that holds a unit: the last one that starts at or before it (one without units starts where its
    // successor does)
    auto sequence_of = [&](int unit) {
        int a = 0, z = geo.batch;
        while (z - a > 1) {
            const int mid = (a + z) >> 1;
            if (first_unit[mid] <= unit) a = mid; else z = mid;
        }
        return a;
    };
    int b = lo < hi ? sequence_of(lo) : 0;
    int first_page = (lo - first_unit[b]) * kUnitPages;
    int entries[kHalfPages / 32];   // block-table entries of one half of the offset table
    auto look_up = [&](int page) {   // of pages [page, page + 128) of sequence b
#pragma unroll
        for (int k = 0; k < kHalfPages / 32; ++k) {
            const int i = page + k * 32 + lane;
            entries[k] = i < geo.max_pages ? ld_ca_s32(block_table + (long long)b * geo.max_pages + i) : -1;
        }
    };
    if (lo < hi) look_up(first_page);

    pdl_launch_dependents();
    if (zero_word && blockIdx.x == 0 && threadIdx.x == 0) *zero_word = 0;
    if (zero_words)
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < zero_count; i += gridDim.x * blockDim.x) zero_words[i] = 0;

    int32_t* off_tab = (int32_t*)(scan_smem + warp * ListCfg<G>::WARP_BYTES);   // in 16-byte units, -1 = no valid page
    const int page_units = geo.kv_heads_stored * (kRowBytes / 16);
    const uint8_t* srow = reinterpret_cast<const uint8_t*>(summaries) + (long long)(g / geo.kv_div) * kRowBytes + c * 16;
    int tab_row[ROWS];   // the table entry of this lane's r-th row of a round
#pragma unroll
    for (int r = 0; r < ROWS; ++r) tab_row[r] = gi * ROWS + (r ^ kr);
    const int own_r = VALS == 16 ? c / G : (c & 7) / G, own_h = c % G;
    const bool owns = VALS == 16 || c < 8;

#pragma unroll 1
    while (lo < hi) {   // one sequence's part of the range
        const int end = min(hi, first_unit[b + 1]);
        const int n_pages = min((end - lo) * kUnitPages, pages_in(b) - first_page);
        const int n_rounds = (n_pages + ROUND_PAGES - 1) / ROUND_PAGES;
        uint4 qraw[G];
#pragma unroll
        for (int hh = 0; hh < G; ++hh)
            qraw[hh] = ld_nc_16B(q + ((long long)b * geo.n_q_heads + g * G + (hh ^ kh)) * kHeadDim + c * 8);
        auto put_half = [&](int half) {
#pragma unroll
            for (int k = 0; k < kHalfPages / 32; ++k) {
                const int i = half * kHalfPages + k * 32 + lane, p = entries[k];
                off_tab[i & (2 * kHalfPages - 1)] = i < n_pages && p >= 0 && p < geo.pool_pages ? p * page_units : -1;
            }
            __syncwarp();
        };
        __syncwarp();   // the table's last reader of the previous part
        put_half(0);
        float* out_lane = scores + ((long long)b * geo.n_q_heads + g * G + own_h) * geo.max_pages + first_page + gi * ROWS + own_r;
        // rows without a valid page and those past the part read row 0 of the pool; their result is never stored
        uint4 rows[DEPTH][ROWS];
        auto fetch = [&](int slot, int R) {
            const int* tab = off_tab + ((R * ROUND_PAGES) & (2 * kHalfPages - 1));
#pragma unroll
            for (int r = 0; r < ROWS; ++r) rows[slot][r] = ld_nc_16B(srow + (long long)max(tab[tab_row[r]], 0) * 16);
        };
#pragma unroll
        for (int t = 0; t < DEPTH; ++t)
            if (t < n_rounds) fetch(t, t);
#pragma unroll 1
        for (int R0 = 0; R0 < n_rounds; R0 += DEPTH) {
            // the table's next half: asked for at the start of this one, stored before the loads reach it
            if (R0 % RPH == 0) look_up(first_page + (R0 / RPH + 1) * kHalfPages);
            if (R0 % RPH == RPH - DEPTH) put_half(R0 / RPH + 1);
#pragma unroll
            for (int t = 0; t < DEPTH; ++t) {
                const int R = R0 + t;
                if (R >= n_rounds) break;
                float vals[16];
#pragma unroll
                for (int r = 0; r < ROWS; ++r)
#pragma unroll
                    for (int hh = 0; hh < G; ++hh) vals[r * G + hh] = chunk_partial_bf16(qraw[hh], rows[t][r]);
                if (R + DEPTH < n_rounds) fetch(t, R + DEPTH);
                float s;
                if constexpr (XOR_MAP) {
                    s = reduce_scatter16_xor(vals);
                } else {
#pragma unroll
                    for (int i = VALS; i < 16; ++i) vals[i] = 0.0f;
                    s = reduce_scatter16(vals, c);
                }
                const int pl = R * ROUND_PAGES + gi * ROWS + own_r;
                if (owns && pl < n_pages) out_lane[R * ROUND_PAGES] = off_tab[pl & (2 * kHalfPages - 1)] >= 0 ? s : -INFINITY;
            }
        }
        lo = end;
        if (lo < hi) {
            b = sequence_of(lo);
            first_page = 0;
            look_up(0);
        }
    }
}

// Exact top-P of one unit's page scores, order (score descending, page ascending).
// KPT > 0: every thread keeps its KPT scores in registers (max_pages <= KPT * blockDim.x);
// KPT == 0: scores staged in shared memory, any size.
template <int KPT>
__global__ void route_select_kernel(Geometry geo, const float* __restrict__ scores,
                                    const int32_t* __restrict__ seq_lens, int P,
                                    int32_t* __restrict__ routed_pages, float* __restrict__ routed_scores,
                                    const int32_t* __restrict__ page_budget)
{
    extern __shared__ uint32_t smem[];
    pdl_wait();
    pdl_launch_dependents();
    const PageSelectSmem s = carve_page_select(smem, geo.max_pages, P);
    const int h = blockIdx.x, b = blockIdx.y;
    const long long unit = (long long)b * geo.n_q_heads + h;
    const int T = seq_lens[b];
    const bool ok = geo.length_ok(T);
    const int n = ok ? geo.pages_of(T) : 0;
    const int P_sel = page_budget ? min(P, __ldcg(page_budget + unit)) : P;   // scored pages only (two-level routing)
    int K;
    if constexpr (KPT > 0)
        K = select_top_pages_reg<KPT>(scores + unit * geo.max_pages, n, P_sel, s);
    else
        K = select_top_pages(scores + unit * geo.max_pages, n, P_sel, s);
    for (int t = threadIdx.x; t < P; t += blockDim.x) {
        routed_pages[unit * P + t] = t < K ? s.win_idx[t] : -1;
        if (routed_scores) routed_scores[unit * P + t] = t < K ? key_to_float(s.win_key[t]) : -INFINITY;
    }
}


size_t select_smem_bytes(const Geometry& g, int P) { return (size_t)select_pages_words(g.max_pages, P) * 4; }

int scan_blocks_per_warp(const Geometry& g)
{
    // 32-page blocks per warp: about one resident wave of warps (2 thread blocks of 8 warps per SM)
    // while that takes no more than kMaxBlocksPerWarp
    const long long blocks = (long long)g.batch * g.n_kv_heads * ((g.max_pages + kBlockPages - 1) / kBlockPages);
    const long long resident_warps = 2LL * kScanWarps * device_sm_count();
    long long k = (blocks + resident_warps - 1) / resident_warps;
    if (k < 1) k = 1;
    if (k > kMaxBlocksPerWarp) k = kMaxBlocksPerWarp;
    return (int)k;
}

// Warps per thread block (8 at most).  When the whole launch is resident at once (two blocks per SM)
// the busiest SM sets the time, so smaller blocks that spread the warps over more SMs
// win: the 64 warps of one 4k-token sequence run as 64 blocks of one warp instead of 8 blocks of 8
// (0.6 us per layer at batch 1); 2048 warps as 296 blocks of 7 instead of 256 of 8.
int scan_warps_per_block(int warps_per_seq, int batch)
{
    const int sms = device_sm_count();
    int best = kScanWarps, best_load = 1 << 30;
    for (int wpb = kScanWarps; wpb >= 1; --wpb) {
        const long long blocks = (long long)batch * ((warps_per_seq + wpb - 1) / wpb);
        if (blocks > 2 * sms) continue;
        const int load = blocks <= sms ? wpb : 2 * wpb;   // warps on the busiest SM
        if (load < best_load) best = wpb, best_load = load;
    }
    return best;
}

template <int G, bool CERT, int D, bool PACKED>
cudaError_t launch_scan_variant(const dim3& grid, int wpb, int bpw, const Geometry& g, const uint16_t* q,
                                const uint16_t* summaries, const int32_t* block_table, const int32_t* seq_lens, float* scores,
                                int32_t* zero_word, int32_t* zero_words, int zero_count, const float* radii,
                                float* rad_logical, cudaStream_t stream)
{
    // The request is padded to 81 KB so that exactly two blocks are resident per SM: with a third one
    // fewer blocks of the kernel that follows fit beside the scan's to start early, and the step gets
    // slower although the scan does not (measured: 30.0 against 24.8 us per layer at batch 8, T = 32k).
    // A grid of no more blocks than SMs, of three warps or more each, asks for so much that no SM takes two (beside the
    // ring of an idle dense block they would pair up: two sequences of 32k tokens 16.1 -> 14.6 us per layer; blocks of
    // one or two warps do not gain).
    const bool spread = wpb >= 3 && (long long)grid.x * grid.y <= device_sm_count();
    const size_t smem = std::max((size_t)kScanWarps * ScanCfg<G, D>::WARP_BYTES, (size_t)(spread ? 120 : 81) * 1024);
    static bool attr_done[kMaxDevices] = {};   // per template instance
    const cudaError_t e = allow_large_dynamic_smem(route_scan_kernel<G, CERT, D, PACKED>, attr_done);
    if (e != cudaSuccess) return e;
    return launch_pdl(route_scan_kernel<G, CERT, D, PACKED>, grid, dim3(wpb * 32), smem, stream, g, q, summaries,
                      block_table, seq_lens, scores, bpw, zero_word, zero_words, zero_count, radii, rad_logical);
}

template <int G, bool CERT, int D = kHeadDim>
cudaError_t launch_scan_g(const Geometry& g, const uint16_t* q, const uint16_t* summaries, const int32_t* block_table,
                          const int32_t* seq_lens, float* scores, int32_t* zero_word, int32_t* zero_words,
                          int zero_count, const float* radii, float* rad_logical, cudaStream_t stream)
{
    if constexpr (!CERT && D == kHeadDim && G != 2) {
        // Share the pages that exist, instead of a grid sized for the longest sequence.  A wave of the grid ends with its
        // slowest warp and each warp pays its start-up; the list pays a longer start and an ordinary launch once, about
        // 3 us.  It wins from so many waves of 32-page blocks on, where the table holds long sequences; microseconds per
        // layer, grid / list, by waves:
        //   four heads a group: 2.2 33 / 36, 3.5 27.7 / 28.8 (4 of 128k) and 39.2 / 39.1 (16 of 32k), 4.3 44.9 / 42.3 (10 of
        //   64k), 5.2 39.7 / 37.1 (6 of 128k) and 62.2 / 61.5 (24 of 32k), 6.9 46.8 / 43.1 (8 of 128k) and 70.9 / 69.4 (32
        //   of 32k), 13.8 79.2 / 75.9 (16 of 128k);
        //   eight, whose round computes twice as long on a row: 1.7 42.1 / 40.0, 2.2 58.3 / 57.2, 3.5 40.6 / 37.8, 13.8 149 / 144;
        //   one: 1.7 19.6 / 20.1, 2.6 22.9 / 23.1, 3.5 25.7 / 26.1, 4.3 33.3 / 29.0, 6.9 37.8 / 35.0, 13.8 68.6 / 58.8;
        //   two: the list loses (6.9 78.2 / 82.2, 104 / 111).
        // Short sequences gain nothing: with four heads 64 of 16k 94.8 / 94.8, 48 of 16k 80.1 / 80.9, 64 of 12k 88.5 / 89.4;
        // with eight 64 of 8k 150 / 150; with one 16 of 8k 40.4 / 41.1.
        // Where the pool has fewer than half of the pages that `batch` sequences of the table's width would have of their own -
        // the sequences are of uneven length, or share prefixes - two waves are enough (lengths are not known here): 64
        // sequences of 4k - 128k with four heads a group 162 / 149, with eight 288 / 253; 32 of 2k - 128k 84.8 / 75.5, with
        // one head a group 149 / 129; 48 of 2k - 32k 86.9 / 86.7.
        // (The sums over the lengths are formed by every block, hence a bound on their number.)
        const long long warps = (long long)g.batch * g.n_kv_heads * ((g.max_pages + kBlockPages - 1) / kBlockPages);
        const long long wave = 2LL * kScanWarps * device_sm_count();
        const bool uneven = (long long)g.batch * g.max_pages >= 2 * g.pool_pages;
        constexpr int kHalfWaves = G == 8 ? 3 : 8;
        const bool enough = (uneven && warps > 2 * wave) ||
                            (g.max_pages >= kListPages && g.batch <= kListBatch && 2 * warps >= kHalfWaves * wave);
        if (!g.super_pages && enough && g.n_kv_heads <= wave) {
            const int ranges = (int)(wave / g.n_kv_heads);
            // (no more than it needs: its loads go to registers, through what shared memory leaves of the L1.  With the 81 KB of the
            // kernel above 16 sequences of 128k take 75.9 us per layer instead of 74.6, 32 of 32k 68.0 instead of 66.9)
            const size_t smem = kScanWarps * (size_t)ListCfg<G>::WARP_BYTES + ((size_t)g.batch + 1) * 4;
            static bool attr_done[kMaxDevices] = {};
            const cudaError_t e = allow_large_dynamic_smem(route_list_kernel<G>, attr_done);
            if (e != cudaSuccess) return e;
            return launch_in_order(route_list_kernel<G>, dim3((unsigned)((ranges * g.n_kv_heads + kScanWarps - 1) / kScanWarps)),
                                   dim3(kScanThreads), smem, stream, g, q, summaries, block_table, seq_lens, scores, ranges,
                                   zero_word, zero_words, zero_count);
        }
    }
    const int bpw = scan_blocks_per_warp(g);
    const int slices = ((g.max_pages + kBlockPages - 1) / kBlockPages + bpw - 1) / bpw;
    const int warps = slices * g.n_kv_heads;
    const int wpb = scan_warps_per_block(warps, g.batch);
    const dim3 grid((unsigned)((warps + wpb - 1) / wpb), (unsigned)g.batch);
    // A grid of one wave is bound by the chain of a warp, longer ones by the FMA pipe: batch 1, T = 4k 0.4 us less with
    // packed rows, batch 8, T = 32k 0.6 us less (one sequence of 128k tokens 0.1 us more); batch 16, T = 128k, several waves, 1.2 us more.
    if ((long long)grid.x * grid.y <= 2LL * device_sm_count())
        return launch_scan_variant<G, CERT, D, true>(grid, wpb, bpw, g, q, summaries, block_table, seq_lens, scores, zero_word,
                                                     zero_words, zero_count, radii, rad_logical, stream);
    return launch_scan_variant<G, CERT, D, false>(grid, wpb, bpw, g, q, summaries, block_table, seq_lens, scores, zero_word,
                                                  zero_words, zero_count, radii, rad_logical, stream);
}

}  // namespace

size_t route_workspace_bytes(const Geometry& g)
{
    return (size_t)g.batch * g.n_q_heads * g.max_pages * sizeof(float);
}

cudaError_t launch_route_scan(const Geometry& g_in, const void* q, const void* summaries, const int32_t* block_table,
                              const int32_t* seq_lens, void* ws, int32_t* zero_word, int32_t* zero_words,
                              int zero_count, cudaStream_t stream, const float* radii, float* rad_logical)
{
    const Geometry g = with_virtual_kv_heads(g_in);
    float* scores = (float*)ws;
    const uint16_t* qq = (const uint16_t*)q;
    const uint16_t* ss = (const uint16_t*)summaries;
#define VSA_SCAN_CASE(G)                                                                                       \
    case G:                                                                                                    \
        if (g.head_dim == 64)                                                                                  \
            return launch_scan_g<G, false, 64>(g, qq, ss, block_table, seq_lens, scores, zero_word, zero_words, \
                                               zero_count, nullptr, nullptr, stream);                          \
        if (g.head_dim == 256)                                                                                 \
            return launch_scan_g<G, false, 256>(g, qq, ss, block_table, seq_lens, scores, zero_word, zero_words, \
                                                zero_count, nullptr, nullptr, stream);                         \
        return radii ? launch_scan_g<G, true>(g, qq, ss, block_table, seq_lens, scores, zero_word, zero_words, \
                                              zero_count, radii, rad_logical, stream)                          \
                     : launch_scan_g<G, false>(g, qq, ss, block_table, seq_lens, scores, zero_word, zero_words, \
                                               zero_count, nullptr, nullptr, stream);
    if (g.head_dim != kHeadDim && radii) return cudaErrorInvalidValue;   // (refused by the entry points)
    switch (g.group) {
        VSA_SCAN_CASE(1)
        VSA_SCAN_CASE(2)
        VSA_SCAN_CASE(4)
        VSA_SCAN_CASE(8)
        default: return cudaErrorInvalidValue;
    }
#undef VSA_SCAN_CASE
}

cudaError_t launch_route_select(const Geometry& g, const void* ws, const int32_t* seq_lens, int P,
                                int32_t* routed_pages, float* routed_scores, cudaStream_t stream,
                                const int32_t* page_budget)
{
    const size_t smem = select_smem_bytes(g, P);
    const dim3 grid((unsigned)g.n_q_heads, (unsigned)g.batch);
#define VSA_SELECT_LAUNCH(KPT, THREADS)                                                                          \
    {                                                                                                            \
        static bool attr_done[kMaxDevices] = {};                                                                 \
        if (smem > 48 * 1024) {                                                                                  \
            const cudaError_t e = allow_large_dynamic_smem(route_select_kernel<KPT>, attr_done);                 \
            if (e != cudaSuccess) return e;                                                                      \
        }                                                                                                        \
        cudaError_t e2 = launch_pdl(route_select_kernel<KPT>, grid, dim3(THREADS), smem, stream, g,            \
                                    (const float*)ws, seq_lens, P, routed_pages, routed_scores, page_budget);  \
        if (e2 != cudaSuccess) return e2;                                                                       \
    }
    if (g.max_pages <= 2048) VSA_SELECT_LAUNCH(8, 256)
    else if (g.max_pages <= 4096) VSA_SELECT_LAUNCH(16, 256)
    else if (g.max_pages <= 8192) VSA_SELECT_LAUNCH(32, 256)
    else VSA_SELECT_LAUNCH(0, 512)
#undef VSA_SELECT_LAUNCH
    return cudaGetLastError();
}

}  // namespace vsa
