// Page summaries: mean of the valid key rows of each page, per KV head (paper Sec. 7 step 1 names
// "coarse page summaries k_page" without defining them; the mean key is this library's reading).
#include "vsa_device.cuh"
#include "vsa_launch.h"

namespace vsa {

// Chunks of 256 threads' work that one block of the summary kernels takes: the grid is sized for the longest
// sequence, and with one chunk per block the blocks past the shorter ones cost 10 us of 120 (8 prompts of 8k - 32k
// tokens, two layers); six waves of blocks (four per SM) stay, so small prompts still spread over the chip and the last
// wave is a small part (three waves: 153.6 against 149.4 us over 32 prompts of 2k - 16k tokens in 32-token pages).
static int summary_chunks(long long threads, int batch)
{
    const long long c = threads * batch / (256LL * 24 * device_sm_count());
    return (int)(c < 1 ? 1 : c > 8 ? 8 : c);
}

// acc[0..8) += a row's eight bf16 values, one rounded fp32 addition each (mixed-precision additions on the packed
// words: no unpacking)
__device__ __forceinline__ void add_row(float (&acc)[8], const uint4& row)
{
    const uint32_t w[4] = {row.x, row.y, row.z, row.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
        asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tadd.rn.f32.bf16 %0, lo, %0;\n\tadd.rn.f32.bf16 %1, hi, %1;\n\t}"
            : "+f"(acc[2 * i]), "+f"(acc[2 * i + 1])
            : "r"(w[i]));
}

// the same for eight e4m3 bytes (exact as f16)
__device__ __forceinline__ void add_row_e4m3(float (&acc)[8], const uint2& row)
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const unsigned short pair = (unsigned short)(((i < 2) ? row.x : row.y) >> (16 * (i & 1)));
        unsigned int h2;
        asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(pair));
        asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tadd.rn.f32.f16 %0, lo, %0;\n\tadd.rn.f32.f16 %1, hi, %1;\n\t}"
            : "+f"(acc[2 * i]), "+f"(acc[2 * i + 1])
            : "r"(h2));
    }
}

// IEEE division by n, round-to-nearest-even to bf16, packed.  For a power of two (every full page) the product with
// its reciprocal is the same correctly rounded value.
__device__ __forceinline__ uint4 mean_to_bf16(const float (&acc)[8], int n)
{
    float m[8];
    const float fn = (float)n;
    if ((n & (n - 1)) == 0) {
        const float r = 1.0f / fn;
#pragma unroll
        for (int e = 0; e < 8; ++e) m[e] = __fmul_rn(acc[e], r);
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) m[e] = __fdiv_rn(acc[e], fn);
    }
    uint4 o;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o.x) : "f"(m[1]), "f"(m[0]));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o.y) : "f"(m[3]), "f"(m[2]));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o.z) : "f"(m[5]), "f"(m[4]));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o.w) : "f"(m[7]), "f"(m[6]));
    return o;
}

// Mean of the first n rows (this thread's 8 columns of each): fp32 sum in ascending token order.
template <int PS>
__device__ __forceinline__ uint4 mean_of_rows(const uint4 (&rows)[PS], int n)
{
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
#pragma unroll
    for (int t = 0; t < PS; ++t)
        if (t < n) add_row(acc, rows[t]);
    return mean_to_bf16(acc, n);
}

// Radius of the first n rows around mu (see radii_kernel), computed by the 16 lanes of a half-warp
// (lane c = columns 8c .. 8c+7, `hmask` = the half-warp's lanes); every lane returns the value.
template <int PS>
__device__ __forceinline__ float radius_of_rows(const uint4 (&rows)[PS], int n, const uint4& mu_bits, int c,
                                                unsigned hmask)
{
    float mu[8];
    unpack8(mu_bits, mu);
    float d2 = 0.0f;   // lane t: the largest |k_t' - mu|^2 over its rows t' = t, t + 16, ...; 0 for absent rows
#pragma unroll
    for (int t0 = 0; t0 < PS; t0 += 16) {
        float vals[16];
#pragma unroll
        for (int t = 0; t < 16; ++t) {
            float f[8], d[8];
            unpack8(rows[t0 + t], f);
#pragma unroll
            for (int e = 0; e < 8; ++e) d[e] = __fsub_rn(f[e], mu[e]);
            vals[t] = t0 + t < n ? chunk_partial(d, d) : 0.0f;
        }
        d2 = fmaxf(d2, reduce_scatter16(vals, c, hmask));
    }
#pragma unroll
    for (int off = 8; off; off >>= 1) d2 = fmaxf(d2, __shfl_xor_sync(hmask, d2, off));
    float m2 = chunk_partial(mu, mu);
#pragma unroll
    for (int off = 8; off; off >>= 1) m2 = m2 + __shfl_xor_sync(hmask, m2, off);
    return __fadd_rn(__fmul_rn(__fsqrt_rn(d2), 1.001f), __fmul_rn(__fsqrt_rn(m2), 0x1p-12f));
}

// One thread per (logical page, kv head, slice of 8 elements): the D / 8 threads of a (page, head) read one
// contiguous key row per load.  fp32 sum in ascending token order, IEEE division by the number of valid rows,
// round-to-nearest-even to bf16.  Bound by HBM: eight rows of a page in flight per thread and four blocks per SM
// keep 128 KB in flight while other blocks add (8 prompts of 8k - 32k tokens, two layers: 112.9 us with three blocks, 103.3
// with four, 109.4 with five; e4m3 64.6 / 57.8 / 66.0).  At four the 64 registers leave 28 bytes of spills (e4m3, 32-token
// pages, 8), which cost less than the fourth block brings; three have none, five more.  Grid: x = chunks of pages, y = sequence.
template <int PS, int D>
__global__ void __launch_bounds__(256, 4) summaries_kernel(Geometry geo, const uint16_t* __restrict__ k_cache,
                                                           const int32_t* __restrict__ block_table,
                                                           const int32_t* __restrict__ seq_lens,
                                                           const int32_t* __restrict__ first_page,
                                                           uint16_t* __restrict__ summaries, int chunks)
{
    constexpr int SL = D / 8;   // slices per row
    pdl_wait();
    pdl_launch_dependents();
    const int b = blockIdx.y;
    const int T = seq_lens[b];
    if (T <= 0 || T > geo.max_pages * PS) return;
    const int nb = (T + PS - 1) / PS;
    const int l0 = first_page ? first_page[b] : 0;
#pragma unroll 1
    for (int chunk = 0; chunk < chunks; ++chunk) {
        const uint32_t idx = (blockIdx.x * chunks + chunk) * 256u + threadIdx.x;   // (2^15 pages * 4096 heads * 32 slices at most)
        const int c = (int)(idx % SL);
        const int g = (int)((idx / SL) % (uint32_t)geo.n_kv_heads);
        const int l = (int)((idx / SL) / (uint32_t)geo.n_kv_heads);
        if (l >= nb) return;
        if (l < l0) continue;
        const long long p = block_table[(long long)b * geo.max_pages + l];
        if (p < 0 || p >= geo.pool_pages) continue;
        const int n = min(PS, T - l * PS);

        const uint16_t* src = k_cache + p * geo.page_stride + (long long)g * geo.head_stride + c * 8;
        float acc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
#pragma unroll 1
        for (int t0 = 0; t0 < n; t0 += 8) {
            uint4 rows[8];
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if (t0 + t < n) rows[t] = ld_nc_16B(src + (long long)(t0 + t) * geo.token_stride);
#pragma unroll
            for (int t = 0; t < 8; ++t)
                if (t0 + t < n) add_row(acc, rows[t]);
        }
        *reinterpret_cast<uint4*>(summaries + (p * geo.n_kv_heads + g) * D + c * 8) = mean_to_bf16(acc, n);
    }
}

// The same for an fp8 cache (e4m3 bytes, value = byte * scale with one scale per page and KV head): the
// decoded bytes are summed in fp32 in ascending token order, multiplied by the scale, divided by the number of
// valid rows and rounded to bf16 - with power-of-two scales bit for bit the summary of the bf16 cache that
// holds the same values.
// One thread per (logical page, kv head, 8-byte slice); head dimension 128.
template <int PS>
__global__ void __launch_bounds__(256, 4) summaries_fp8_kernel(Geometry geo, const uint8_t* __restrict__ k_cache,
                                                               const float* __restrict__ k_scale,
                                                               const int32_t* __restrict__ block_table,
                                                               const int32_t* __restrict__ seq_lens,
                                                               const int32_t* __restrict__ first_page,
                                                               uint16_t* __restrict__ summaries, int chunks)
{
    constexpr int SL = kHeadDim / 8;   // slices per row
    pdl_wait();
    pdl_launch_dependents();
    const int b = blockIdx.y;
    const int T = seq_lens[b];
    if (T <= 0 || T > geo.max_pages * PS) return;
    const int nb = (T + PS - 1) / PS;
    const int l0 = first_page ? first_page[b] : 0;
#pragma unroll 1
    for (int chunk = 0; chunk < chunks; ++chunk) {
        const uint32_t idx = (blockIdx.x * chunks + chunk) * 256u + threadIdx.x;   // (2^15 pages * 4096 heads * 32 slices at most)
        const int c = (int)(idx % SL);
        const int g = (int)((idx / SL) % (uint32_t)geo.n_kv_heads);
        const int l = (int)((idx / SL) / (uint32_t)geo.n_kv_heads);
        if (l >= nb) return;
        if (l < l0) continue;
        const long long p = block_table[(long long)b * geo.max_pages + l];
        if (p < 0 || p >= geo.pool_pages) continue;
        const int n = min(PS, T - l * PS);

        const uint8_t* src = k_cache + p * geo.page_stride + (long long)g * geo.head_stride + c * 8;
        const float scale = __ldg(k_scale + p * geo.n_kv_heads + g);
        float acc[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
#pragma unroll 1
        for (int t0 = 0; t0 < n; t0 += 16) {
            uint2 rows[16];
#pragma unroll
            for (int t = 0; t < 16; ++t)
                if (t0 + t < n) rows[t] = ld_nc_8B(src + (long long)(t0 + t) * geo.token_stride);
#pragma unroll
            for (int t = 0; t < 16; ++t)
                if (t0 + t < n) add_row_e4m3(acc, rows[t]);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = __fmul_rn(acc[e], scale);
        *reinterpret_cast<uint4*>(summaries + (p * geo.n_kv_heads + g) * kHeadDim + c * 8) = mean_to_bf16(acc, n);
    }
}

// Radius of each page around its stored summary (the ball bound of the routing certificate):
//   rhat = 1.001 * sqrt(max_t |k_t - mu|^2) + 2^-12 * |mu|,
// squared norms summed in the library's canonical order, every operation a single rounded fp32
// operation so that the CPU oracle reproduces the value bit for bit.  Same thread mapping as the
// summaries kernel; the 16 threads of a (page, head) form a half-warp and only talk to each other.
template <int PS>
__global__ void __launch_bounds__(256) radii_kernel(Geometry geo, const uint16_t* __restrict__ k_cache,
                                                    const uint16_t* __restrict__ summaries,
                                                    const int32_t* __restrict__ block_table,
                                                    const int32_t* __restrict__ seq_lens,
                                                    const int32_t* __restrict__ first_page,
                                                    float* __restrict__ radii)
{
    const int b = blockIdx.y;
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = (int)(idx & 15);
    const int g = (int)((idx >> 4) % geo.n_kv_heads);
    const long long l = (idx >> 4) / geo.n_kv_heads;
    const int T = seq_lens[b];
    if (T <= 0 || T > geo.max_pages * PS) return;
    const int nb = (T + PS - 1) / PS;
    const int l0 = first_page ? first_page[b] : 0;
    if (l < l0 || l >= nb) return;
    const long long p = block_table[(long long)b * geo.max_pages + l];
    if (p < 0 || p >= geo.pool_pages) return;
    const int n = min(PS, T - (int)l * PS);
    const unsigned hmask = 0xffffu << (threadIdx.x & 16);   // this half-warp (the other may have returned)

    const uint4 mu_bits = *reinterpret_cast<const uint4*>(summaries + (p * geo.n_kv_heads + g) * kHeadDim + c * 8);
    const uint16_t* src = k_cache + p * geo.page_stride + (long long)g * geo.head_stride + c * 8;
    uint4 rows[PS];
#pragma unroll
    for (int t = 0; t < PS; ++t)
        rows[t] = t < n ? ld_nc_16B(src + (long long)t * geo.token_stride) : make_uint4(0u, 0u, 0u, 0u);
    const float rhat = radius_of_rows<PS>(rows, n, mu_bits, c, hmask);
    if (c == 0) radii[p * geo.n_kv_heads + g] = rhat;
}

// Appends one token per sequence to the paged cache and brings the page it lands in up to date: its
// key and value rows, the page's summary and (when asked for) its radius.  A half-warp per
// (sequence, kv head); seq_lens are the lengths AFTER the append.
template <int PS>
__global__ void __launch_bounds__(256) append_kernel(Geometry geo, const uint16_t* __restrict__ k_new,
                                                     const uint16_t* __restrict__ v_new, uint16_t* __restrict__ k_cache,
                                                     uint16_t* __restrict__ v_cache,
                                                     const int32_t* __restrict__ block_table,
                                                     const int32_t* __restrict__ seq_lens,
                                                     uint16_t* __restrict__ summaries, float* __restrict__ radii)
{
    // Launched with programmatic serialisation like the kernels of the step, so that neither side of it pays a full
    // launch gap (0.8 us of a 16 us layer at batch 1).  What bounds it is a chain of loads: length, table entry, rows.  So the
    // length and the entry are read once ahead of the wait, when they may still be about to change, and only to know where
    // the page probably is: its rows are asked for in L2, and after the wait everything is read (again) at once.  Where the
    // length or the entry did change, the chain is walked as it is.
    const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = (int)(idx & 15);
    const long long pair = idx >> 4;
    if (pair >= (long long)geo.batch * geo.n_kv_heads) return;
    const int b = (int)(pair / geo.n_kv_heads), g = (int)(pair % geo.n_kv_heads);
    const unsigned hmask = 0xffffu << (threadIdx.x & 16);
    const int32_t* bt = block_table + (long long)b * geo.max_pages;
    auto length_ok = [&](int T) { return T > 0 && T <= geo.max_pages * PS; };
    auto page_ok = [&](long long p) { return p >= 0 && p < geo.pool_pages; };
    const int T0 = ld_cg_s32(seq_lens + b), l0 = length_ok(T0) ? (T0 - 1) / PS : 0;
    const long long p0 = ld_cg_s32(bt + l0);
    const bool expected = length_ok(T0) && page_ok(p0);
    const long long head_off = (long long)g * geo.head_stride + c * 8;
    if (expected) {
        const uint16_t* page = k_cache + p0 * geo.page_stride + (long long)g * geo.head_stride;
        for (int t = c; t < (T0 - 1) % PS; t += 16) {
            prefetch_L2(page + (long long)t * geo.token_stride);
            prefetch_L2(page + (long long)t * geo.token_stride + kHeadDim / 2);
        }
    }

    pdl_wait();
    pdl_launch_dependents();
    int T = ld_cg_s32(seq_lens + b);
    long long p = ld_cg_s32(bt + l0);
    const uint4 kn = ld_cg_16B(k_new + pair * kHeadDim + c * 8);
    const uint4 vn = ld_cg_16B(v_new + pair * kHeadDim + c * 8);
    uint4 rows[PS];
    auto fetch = [&](long long page, int n) {   // the rows before the new one
#pragma unroll
        for (int t = 0; t < PS; ++t)
            rows[t] = t < n - 1 ? ld_cg_16B(k_cache + page * geo.page_stride + head_off + (long long)t * geo.token_stride)
                                : make_uint4(0u, 0u, 0u, 0u);
    };
    if (expected) fetch(p0, (T0 - 1) % PS + 1);
    if (!expected || T != T0 || p != p0) {
        if (!length_ok(T)) return;
        p = ld_cg_s32(bt + (T - 1) / PS);
        if (!page_ok(p)) return;
        fetch(p, (T - 1) % PS + 1);
    }
    __syncwarp(hmask);

    const int n = (T - 1) % PS + 1;   // rows that the page holds now
    *reinterpret_cast<uint4*>(k_cache + p * geo.page_stride + head_off + (long long)(n - 1) * geo.token_stride) = kn;
    *reinterpret_cast<uint4*>(v_cache + p * geo.page_stride + head_off + (long long)(n - 1) * geo.token_stride) = vn;
#pragma unroll
    for (int t = 0; t < PS; ++t)
        if (t == n - 1) rows[t] = kn;
    const uint4 mu_bits = mean_of_rows<PS>(rows, n);
    *reinterpret_cast<uint4*>(summaries + (p * geo.n_kv_heads + g) * kHeadDim + c * 8) = mu_bits;
    if (radii) {
        const float rhat = radius_of_rows<PS>(rows, n, mu_bits, c, hmask);
        if (c == 0) radii[p * geo.n_kv_heads + g] = rhat;
    }
}

cudaError_t launch_append(const Geometry& g, const void* k_new, const void* v_new, void* k_cache, void* v_cache,
                          const int32_t* block_table, const int32_t* seq_lens, void* summaries, float* radii,
                          cudaStream_t stream)
{
    // small blocks: a half-warp is a latency chain of four loads, and one warp per SM runs it fastest
    const long long threads = (long long)g.batch * g.n_kv_heads * 16;
    return launch_pdl(g.page_size == 32 ? append_kernel<32> : append_kernel<16>, dim3((unsigned)((threads + 31) / 32)),
                      dim3(32), 0, stream, g, (const uint16_t*)k_new, (const uint16_t*)v_new, (uint16_t*)k_cache,
                      (uint16_t*)v_cache, block_table, seq_lens, (uint16_t*)summaries, radii);
}

cudaError_t launch_build_radii(const Geometry& g, const void* k_cache, const void* summaries,
                               const int32_t* block_table, const int32_t* seq_lens, const int32_t* first_page,
                               float* radii, cudaStream_t stream)
{
    const long long threads = (long long)g.max_pages * g.n_kv_heads * 16;
    dim3 grid((unsigned)((threads + 255) / 256), (unsigned)g.batch);
    auto* kernel = g.page_size == 32 ? radii_kernel<32> : radii_kernel<16>;
    kernel<<<grid, 256, 0, stream>>>(g, (const uint16_t*)k_cache, (const uint16_t*)summaries, block_table,
                                           seq_lens, first_page, radii);
    return cudaGetLastError();
}

cudaError_t launch_build_summaries(const Geometry& g, const void* k_cache, const int32_t* block_table,
                                   const int32_t* seq_lens, const int32_t* first_page, void* summaries,
                                   cudaStream_t stream)
{
    const long long threads = (long long)g.max_pages * g.n_kv_heads * (g.head_dim / 8);
    const int chunks = summary_chunks(threads, g.batch);
    dim3 grid((unsigned)((threads + 256 * chunks - 1) / (256 * chunks)), (unsigned)g.batch);
    auto* kernel = g.page_size == 32 ? summaries_kernel<32, 128> : summaries_kernel<16, 128>;
    if (g.head_dim == 64) kernel = g.page_size == 32 ? summaries_kernel<32, 64> : summaries_kernel<16, 64>;
    if (g.head_dim == 256) kernel = g.page_size == 32 ? summaries_kernel<32, 256> : summaries_kernel<16, 256>;
    return launch_pdl(kernel, grid, dim3(256), 0, stream, g, (const uint16_t*)k_cache, block_table, seq_lens,
                      first_page, (uint16_t*)summaries, chunks);
}

cudaError_t launch_build_summaries_fp8(const Geometry& g, const void* k_cache, const float* k_scale,
                                       const int32_t* block_table, const int32_t* seq_lens,
                                       const int32_t* first_page, void* summaries, cudaStream_t stream)
{
    const long long threads = (long long)g.max_pages * g.n_kv_heads * 16;
    const int chunks = summary_chunks(threads, g.batch);
    dim3 grid((unsigned)((threads + 256 * chunks - 1) / (256 * chunks)), (unsigned)g.batch);
    auto* kernel = g.page_size == 32 ? summaries_fp8_kernel<32> : summaries_fp8_kernel<16>;
    return launch_pdl(kernel, grid, dim3(256), 0, stream, g, (const uint8_t*)k_cache, k_scale, block_table, seq_lens,
                      first_page, (uint16_t*)summaries, chunks);
}

}  // namespace vsa
