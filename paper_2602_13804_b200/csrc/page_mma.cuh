// Page scores on the tensor cores.
//
// The step needs the SET of the P best pages of a query head and their order, not their scores, and both are defined by fp32 sums
// in one fixed order (chunk_partial and the halving tree).  An MMA forms the same dot products with a rounding of its own, and
// A = sum |q_i k_i| beside them bounds the difference: scores further apart than page_score_slack() are in the order of
// the fixed-order ones.  The sparse pass selects by the MMA scores and forms the fixed-order scores of the few pages that
// are closer (sparse_step.cuh), so the routed pages are bit for bit those of a fixed-order scan.
//
// A fixed-order scan issues about 36 warp instructions for a row of 256 bytes and four heads, twice that for eight; here 16 rows
// against up to eight heads take sixteen MMAs and about 110 instructions.
#pragma once

#include "vsa_device.cuh"

namespace vsa {

// How far apart two page scores by MMAs have to be to be told apart, from A >= sum |q_i k_i| of the pages concerned.
// The model: an MMA of depth 16 aligns its exact products to the largest of them and drops what lies more than 24 bits below its top
// (Fasi, Higham, Mikaitis and Pranesh, "Numerical behavior of NVIDIA tensor cores", 2021): with the normalisation its error is
// at most 17 * 2^-23 of its share of A, 19 * 2^-23 if it takes two steps of depth 8.  Adding up D / 16 of them in fp32 costs at
// most 3.5 * 2^-23 A (7.5 at D = 256), the fixed order's own rounding 4 (4.5): 31 in all.  40 covers them, and A's own rounding;
// the slack is twice that, since both scores can be off.  The constant covers sums below the normal range.
// The paper's chips are older ones; that a B200 does no worse is measured, not specified.  Against fp64, 262 thousand scores each of normal
// values, magnitudes spread over 2^32, the same with all mantissa bits set, and pairs that cancel: at most 2.4 * 2^-23 A at D = 64, 2.9 at
// 128, 3.7 at 256, and A itself low by at most 5, 8 and 14 * 2^-23 of it.
__device__ __forceinline__ float page_score_slack(float a) { return a * (80.0f * 1.1920929e-7f) + 1e-30f; }

// From A = 2^126 on, infinities and NaN among them, a sum may overflow in one order and not in another: the page's score is a
// mark, NaN, its A does not count for the bound of the others, and the sparse pass forms its fixed-order score.  (One such
// key in a sequence otherwise has its blocks score every page anew: 64 sequences of 4k - 128k, eight heads a group 853 us, 8 of
// 32k 49, against 294 and 22 without.)
constexpr uint32_t kNoBound = 0x7e800000u;
__device__ __forceinline__ void mark_without_bound(float& score, uint32_t& a)
{
    if (a >= kNoBound) score = __int_as_float(0x7fffffff), a = 0u;
}

namespace {

// D (16x8, fp32) += A (16x16, bf16, row) * B (16x8, bf16, col)
__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the same without a sum to add to
__device__ __forceinline__ void mma_16816_first(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.0f));
}
// the magnitudes of two bf16 (of the query: formed anew for every tile, the registers that kept them would be those of loads in flight)
__device__ __forceinline__ uint32_t abs2(uint32_t x) { return x & 0x7fff7fffu; }
__device__ __forceinline__ uint32_t abs2_here(uint32_t x)
{
    uint32_t r;
    asm volatile("and.b32 %0, %1, 0x7fff7fff;" : "=r"(r) : "r"(x));
    return r;
}

// 16 summary rows as A fragments.  Lane (r, j) = (lane / 4, lane % 4) holds 16-byte chunks j, j + 4, ... of rows r and r + 8, and
// of query head r: the halves of a chunk are the fragments of two MMAs (which elements an MMA's index k stands for is the
// same for both operands, so any assignment gives the dot product).
template <int D>
struct PageTile {
    static constexpr int KC = D / 32;   // chunks of a row per lane
    uint4 row[2][KC];

    // s: scores of (row r, head 2 j), (r, 2 j + 1), (r + 8, 2 j), (r + 8, 2 j + 1); a: the sums of the products' magnitudes.  Every
    // MMA of the scores starts from zero and its result is added in fp32: a chain of D / 16 would lose D / 16 times as much
    // as an MMA does (each drops bits relative to the whole sum so far), and as many more pages would be too close to tell.
    __device__ __forceinline__ void dot(const uint4 (&q)[KC], float (&s)[4], float (&a)[4]) const
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) s[i] = 0.0f;
        float a2[4];   // (two chains)
#pragma unroll
        for (int i = 0; i < KC; ++i) {
            float u[4], v[4];
            const uint4 &x = row[0][i], &y = row[1][i];
            mma_16816_first(u, x.x, y.x, x.y, y.y, q[i].x, q[i].y);
            if (i == 0) {
                mma_16816_first(a, abs2(x.x), abs2(y.x), abs2(x.y), abs2(y.y), abs2_here(q[i].x), abs2_here(q[i].y));
            } else {
                mma_16816(a, abs2(x.x), abs2(y.x), abs2(x.y), abs2(y.y), abs2_here(q[i].x), abs2_here(q[i].y));
            }
            mma_16816_first(v, x.z, y.z, x.w, y.w, q[i].z, q[i].w);
            if (i == 0) {
                mma_16816_first(a2, abs2(x.z), abs2(y.z), abs2(x.w), abs2(y.w), abs2_here(q[i].z), abs2_here(q[i].w));
            } else {
                mma_16816(a2, abs2(x.z), abs2(y.z), abs2(x.w), abs2(y.w), abs2_here(q[i].z), abs2_here(q[i].w));
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) s[e] = (s[e] + u[e]) + v[e];
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) a[e] += a2[e];
    }
};

}  // namespace

}  // namespace vsa
