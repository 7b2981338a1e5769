// Page scan of the decode step on the tensor cores, where the scan is several waves of blocks: scores by MMAs and the bound of
// their rounding (page_mma.cuh), for a sparse pass that settles near ties itself.
//
// The 32-page blocks of all sequences form one list that one wave of warps shares evenly, as in route_list_kernel (route.cu); warp w
// takes KV head w % n_kv and the (w / n_kv)-th range of the list, part by part as it crosses sequences.  Two tiles of 16
// rows (D = 64: 2 KB each, 128: 4 KB) of a warp are in flight in registers.  Launched in stream order and without shared memory to
// speak of: loads into registers need lines of the L1, and blocks that start early beside those of the kernels around it run with what
// these leave, 28 KB (16 sequences of 128k 126 us per layer against 74).
// Bound by memory: 16 sequences of 128k, 268 MB of rows, 54.8 -> 50.0 us alone (about 5 of it the start, the chain from the lengths
// to the rows, then 6.3 TB/s); eight heads a group, whose fixed-order scan was bound by its arithmetic, 64 sequences of 4k - 128k
// 89.9 -> 59.4.  Built and slower: whole rows by cp.async and ldmatrix (55), by one bulk copy each (75: 20 cycles a copy on an SM),
// the warps of the eight KV heads in lockstep (no change), the 32-page blocks as a grid (73).
#include <math.h>

#include "page_mma.cuh"
#include "vsa_launch.h"

namespace vsa {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kBlock = kBoundPages;   // pages that a warp handles at a time, and that share one bound

template <int D>
__global__ void __launch_bounds__(kThreads, 2)
mma_list_kernel(Geometry geo, const uint16_t* __restrict__ q, const uint16_t* __restrict__ summaries, const int32_t* __restrict__ block_table,
                const int32_t* __restrict__ seq_lens, float* __restrict__ scores, uint32_t* __restrict__ bounds, int ranges,
                int32_t* zero_word, int32_t* zero_words, int zero_count)
{
    constexpr int KC = PageTile<D>::KC;
    extern __shared__ __align__(16) int32_t first_unit[];   // [batch + 1] first block of every sequence
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r = lane >> 2, j = lane & 3;
    const int w = blockIdx.x * kWarps + warp, g = w % geo.n_kv_heads, range = w / geo.n_kv_heads;
    auto pages_in = [&](int b) {   // 0 for an invalid length
        const int T = ld_ca_s32(seq_lens + b);
        return geo.length_ok(T) ? geo.pages_of(T) : 0;
    };
    // Every warp sums up its own part of the batch (one warp alone takes 0.3 us for 32 sequences), then adds what lies before it.
    {
        __shared__ int warp_units[kWarps];
        const int part = (geo.batch + kThreads - 1) / kThreads * 32, end = min((warp + 1) * part, geo.batch);
        int base = 0;
        for (int b0 = warp * part; b0 < end; b0 += 32) {
            const int u = b0 + lane < end ? (pages_in(b0 + lane) + kBlock - 1) / kBlock : 0;
            int incl = u;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int o = __shfl_up_sync(kFullMask, incl, off);
                if (lane >= off) incl += o;
            }
            if (b0 + lane < end) first_unit[b0 + lane] = base + incl - u;
            base += __shfl_sync(kFullMask, incl, 31);
        }
        if (lane == 0) warp_units[warp] = base;
        __syncthreads();
        int before = 0;
        for (int i = 0; i < warp; ++i) before += warp_units[i];
        for (int i = warp * part + lane; i < end; i += 32) first_unit[i] += before;
        if (warp == kWarps - 1 && lane == 0) first_unit[geo.batch] = before + base;
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
    int first = (lo - first_unit[b]) * kBlock;
    auto look_up = [&](int page, int end) {   // this lane's page of the block at `page` in the pool, -1 if there is none
        const int i = page + lane;
        const int e = i < end ? ld_ca_s32(block_table + (long long)b * geo.max_pages + i) : -1;
        return e >= 0 && e < geo.pool_pages ? e : -1;
    };
    if (zero_word && blockIdx.x == 0 && threadIdx.x == 0) *zero_word = 0;
    if (zero_words)
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < zero_count; i += gridDim.x * blockDim.x) zero_words[i] = 0;
    pdl_launch_dependents();

    const uint8_t* rows = reinterpret_cast<const uint8_t*>(summaries) + (long long)(g / geo.kv_div) * (2 * D) + j * 16;
    const unsigned page_bytes = (unsigned)(geo.kv_heads_stored * 2 * D);
    const bool has0 = 2 * j < geo.group, has1 = 2 * j + 1 < geo.group;
    PageTile<D> tiles[2];
    auto load = [&](int t, int entry) {   // tile t of a block (no valid page: row 0 of the pool, whose result is not used)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = max(__shfl_sync(kFullMask, entry, t * 16 + h * 8 + r), 0);
            const uint8_t* row = rows + (unsigned long long)(unsigned)e * page_bytes;
#pragma unroll
            for (int i = 0; i < KC; ++i) tiles[t].row[h][i] = ld_nc_16B(row + 64 * i);
        }
    };
#pragma unroll 1
    while (lo < hi) {   // one sequence's part of the range
        const int units = min(hi, first_unit[b + 1]) - lo, end = min(first + units * kBlock, pages_in(b));
        int entry = look_up(first, end), next_entry = look_up(first + kBlock, end);
        const uint16_t* q_row = q + ((long long)b * geo.n_q_heads + g * geo.group + r) * D + j * 8;
        uint4 qf[KC];   // (zero where the group has fewer than eight heads)
#pragma unroll
        for (int i = 0; i < KC; ++i) qf[i] = r < geo.group ? ld_nc_16B(q_row + 32 * i) : make_uint4(0u, 0u, 0u, 0u);
        float* out = scores + ((long long)b * geo.n_q_heads + g * geo.group + 2 * j) * geo.max_pages;
        uint32_t* bound = bounds + ((long long)b * geo.n_kv_heads + g) * bound_blocks(geo.max_pages);
        load(0, entry);
        load(1, entry);
#pragma unroll 1
        for (int page = first; page < end; page += kBlock) {
            const int after = look_up(page + 2 * kBlock, end);
            uint32_t most = 0u;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                float s[4], a[4];
                tiles[t].dot(qf, s, a);
                if (page + kBlock < end) load(t, next_entry);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int l = t * 16 + h * 8 + r;
                    const bool ok = __shfl_sync(kFullMask, entry, l) >= 0;
                    // (magnitudes are not negative: their order is that of their bits, an infinity or NaN above all)
                    uint32_t a0 = __float_as_uint(a[2 * h]), a1 = __float_as_uint(a[2 * h + 1]);
                    if (max(a0, a1) >= kNoBound) mark_without_bound(s[2 * h], a0), mark_without_bound(s[2 * h + 1], a1);
                    if (ok) most = max(most, max(a0, a1));
                    if (page + l < end) {
                        if (has0) out[page + l] = ok ? s[2 * h] : -INFINITY;
                        if (has1) out[geo.max_pages + page + l] = ok ? s[2 * h + 1] : -INFINITY;
                    }
                }
            }
            most = __reduce_max_sync(kFullMask, most);
            if (lane == 0) bound[page / kBlock] = most;
            entry = next_entry;
            next_entry = after;
        }
        lo += units;
        if (lo < hi) {
            b = sequence_of(lo);
            first = 0;
        }
    }
}

template <int D>
cudaError_t launch_mma(const Geometry& g, const void* q, const void* summaries, const int32_t* block_table, const int32_t* seq_lens,
                       float* scores, uint32_t* bounds, int32_t* zero_word, int32_t* zero_words, int zero_count, cudaStream_t stream)
{
    const int wave = 2 * kWarps * device_sm_count(), ranges = g.n_kv_heads < wave ? wave / g.n_kv_heads : 1;
    return launch_in_order(mma_list_kernel<D>, dim3((unsigned)((ranges * g.n_kv_heads + kWarps - 1) / kWarps)), dim3(kThreads),
                           ((size_t)g.batch + 1) * 4, stream, g, (const uint16_t*)q, (const uint16_t*)summaries, block_table, seq_lens,
                           scores, bounds, ranges, zero_word, zero_words, zero_count);
}

}  // namespace

size_t route_bound_bytes(const Geometry& g_in)
{
    const Geometry g = with_virtual_kv_heads(g_in);
    return (size_t)g.batch * g.n_kv_heads * bound_blocks(g.max_pages) * 4;
}

// The list pays its start and an ordinary launch, and the sparse pass the bounds and near ties: it wins for tables of 1024 pages and
// more, with four heads a group, whose fixed-order scan needs 0.6 of the issue slots and little more than the time of its bytes, from 4096.
// One head a group never at D = 128, where the fixed-order scan has the least arithmetic.  Microseconds per layer, fixed order / MMA.
// Eight heads: 8 of 16k 30.7 / 28.7, of 32k 35.4 / 32.2, of 64k 54.7 / 49.4, 16 of 16k 55.1 / 53.1, 64 of 16k 169 / 157, 64 of 4k - 128k
// 321 / 301, 20 of 1k - 64k 67.8 / 68.0, 16 heads of one KV head 64 of 64k 146 / 130; shorter 32 of 8k 84.2 / 85.5.  Two: 40 of 16k
// 49.8 / 46.4, 40 of 2k - 64k 54.6 / 48.2.  Four: 16 of 128k 75.6 / 74.3, 12 of 128k 65.2 / 61.6, 10 of 64k 41.1 / 40.0, 24 of 64k
// 78.1 / 78.5, e4m3 cache 16 of 64k 49.3 / 48.3; shorter 10 of 48k 36.7 / 36.8, 32 of 32k 67.3 / 67.3, 48 of 2k - 32k 74.4 / 76.2.  One:
// 32 heads, 16 of 64k 111 / 122.  D = 64 (no list of its own): 16 of 64k 56.8 / 41.3, one head a group 12 of 64k 76.8 / 57.2, eight
// 24 of 64k 214 / 175, 32 of 16k 53.1 / 50.4; shorter 64 of 8k 69.5 / 69.2.  D = 256 gains nothing (16 of 64k 89.3 / 88.5, 32 of 8k 74.6 / 80.8).
bool route_mma_wins(const Geometry& g)
{
    if (g.head_dim == 256 || (g.head_dim == kHeadDim && g.group == 1)) return false;
    return g.max_pages >= (g.head_dim == kHeadDim && g.group == 4 ? 4096 : 1024);
}

cudaError_t launch_route_mma(const Geometry& g_in, const void* q, const void* summaries, const int32_t* block_table, const int32_t* seq_lens,
                             float* scores, uint32_t* bounds, int32_t* zero_word, int32_t* zero_words, int zero_count, cudaStream_t stream)
{
    const Geometry g = with_virtual_kv_heads(g_in);
    if (g.group > 8) return cudaErrorInvalidValue;
    if (g.head_dim == 64) return launch_mma<64>(g, q, summaries, block_table, seq_lens, scores, bounds, zero_word, zero_words, zero_count, stream);
    if (g.head_dim == kHeadDim)
        return launch_mma<kHeadDim>(g, q, summaries, block_table, seq_lens, scores, bounds, zero_word, zero_words, zero_count, stream);
    return cudaErrorInvalidValue;
}

}  // namespace vsa
