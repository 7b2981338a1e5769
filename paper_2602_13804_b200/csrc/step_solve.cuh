// Iterative weights on the candidate set of one unit (step 3 of Sec. 7; Sec. 5.3, App. E): entropic mirror descent
// (SOLVE 1) or Frank-Wolfe with exact line search (SOLVE 2), by the 256 threads of the fused kernel's block.
// Thread j owns candidate j: its score, log-weight and gradient entry live in registers; the candidates' key rows lie
// in shared memory, 256 bytes each, 16-byte chunks XOR-swizzled by the row.
//
// A pass of the descent is y = sum_i a_i k_i followed by g_i = <k_i, y> - s_i, two products of the 64 KB of keys with a
// vector, fp32 on the floating-point pipe; half of the unpacking runs there too, as mixed-precision additions.  Bound by
// the instructions of the passes and by shared-memory bandwidth (two blocks read 256 KB a pass).  Four iterations at
// batch 8, T = 32k: 41.0 -> 37.2 us per layer.  The same products on the tensor cores (the vector as three bf16 columns,
// which is exact) took 41.6: a warp-level MMA costs about twelve cycles and an ldmatrix the bandwidth of these loads.
// Frank-Wolfe picks vertices, integers that the CPU oracle mirrors bit for bit, so it keeps the canonical fp32 order.
#pragma once

#include "vsa_device.cuh"
#include "vsa_launch.h"

namespace vsa {

namespace {

// row r, 16-byte chunk c of the key tile
__device__ __forceinline__ uint32_t tile_at(int r, int c) { return (uint32_t)(r * kRowBytes + ((c ^ (r & 7)) << 4)); }

struct SolveSmem {
    uint8_t* tile;       // key rows of the candidates, zero rows up to a multiple of 32
    uint32_t* stat;      // 80 words of statistics
    float* red;          // [8][128] partial readouts
    float* y;            // [128] readout
    float* weights;      // [256] exchanged inside a warp
};

// Entropic mirror descent.  Returns this candidate's unnormalised weight; lse: log-sum-exp of the closed form.
__device__ __forceinline__ float solve_entropic(const SolveSmem& sm, int ns, float s_own, int iters, float epsilon,
                                                const uint4& q, float& lse, vsa_solve_t* solve)
{
    constexpr int WARPS = 8;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = lane & 15, gi = lane >> 4;
    const bool have = tid < ns, busy = warp * 32 < ns;   // busy: this warp owns a candidate
    float* stat_f = reinterpret_cast<float*>(sm.stat);   // [0..8) partial sums, [8..16) maxima
    const uint8_t* rows = sm.tile + (warp * 32 + gi * 16) * kRowBytes;   // the sixteen rows of this half-warp
    auto row = [&](int r) { return *reinterpret_cast<const uint4*>(rows + tile_at(r, c)); };
    float vals[16];
    // step: eta = 1 / max_i |k_i|^2
    uint32_t lkey = 0u;
    if (busy) {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const uint4 x = row(r);
            vals[r] = chunk_partial_bf16(x, x);
        }
        const float nrm = reduce_scatter16(vals, c);
        lkey = __reduce_max_sync(kFullMask, have ? float_to_key(nrm) : 0u);
    }
    if (lane == 0) sm.stat[16 + warp] = lkey;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < WARPS; ++w) lkey = max(lkey, sm.stat[16 + w]);
    const float Lmax = lkey != 0u ? key_to_float(lkey) : 0.0f;
    const float eta = Lmax > 0.0f ? 1.0f / Lmax : 0.0f;
    const float shrink = 1.0f / (1.0f + eta * epsilon);
    float l_own = have ? s_own / epsilon : -INFINITY;
    float m = 0.0f, Z = 1.0f, a_own = 0.0f, g_own = 0.0f;
    float* my_weights = sm.weights + warp * 32 + gi * 16;
#pragma unroll 1
    for (int it = 0;; ++it) {
        // ---- this warp's part of sum_i e_i k_i, relative to its own maximum ----
        const float mw = key_to_float(__reduce_max_sync(kFullMask, float_to_key(l_own)));
        const float e_own = have ? __expf(l_own - mw) : 0.0f;
        if (busy) {
            my_weights[c] = e_own;
            __syncwarp();
            float ya[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) ya[e] = 0.0f;
#pragma unroll
            for (int r4 = 0; r4 < 16; r4 += 4) {
                const float4 w4 = *reinterpret_cast<const float4*>(my_weights + r4);
                const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    float uf[8];
                    unpack8_mixed(row(r4 + r), uf);
#pragma unroll
                    for (int e = 0; e < 8; e += 2) fma2(ya[e], ya[e + 1], w[r], w[r], uf[e], uf[e + 1]);
                }
            }
            float zw = e_own;
#pragma unroll
            for (int off = 16; off; off >>= 1) zw += __shfl_xor_sync(kFullMask, zw, off);
#pragma unroll
            for (int e = 0; e < 8; ++e) ya[e] += __shfl_xor_sync(kFullMask, ya[e], 16);
            if (gi == 0) {
                float4* dst = reinterpret_cast<float4*>(sm.red + warp * kHeadDim + c * 8);
                dst[0] = make_float4(ya[0], ya[1], ya[2], ya[3]);
                dst[1] = make_float4(ya[4], ya[5], ya[6], ya[7]);
                if (c == 0) {
                    stat_f[warp] = zw;
                    stat_f[8 + warp] = mw;
                }
            }
        } else if (lane == 0) {
            stat_f[warp] = 0.0f;
            stat_f[8 + warp] = -INFINITY;
        }
        __syncthreads();
        // ---- the block's readout: the sums of the warps, rescaled to the common maximum ----
        float f[WARPS];
        m = -INFINITY;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) m = fmaxf(m, stat_f[8 + w]);
        Z = 0.0f;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            f[w] = __expf(stat_f[8 + w] - m);   // 0 for a warp without candidates
            Z = fmaf(stat_f[w], f[w], Z);
        }
        if (tid < kHeadDim) {
            float y = 0.0f;
#pragma unroll
            for (int w = 0; w < WARPS; ++w)
                if (w * 32 < ns) y = fmaf(f[w], sm.red[w * kHeadDim + tid], y);
            sm.y[tid] = y * (1.0f / Z);
        }
        __syncthreads();
        a_own = have ? e_own * __expf(mw - m) : 0.0f;   // exp(l_own - m)
        // ---- gradient of the quadratic part: g_i = <k_i, y> - <k_i, q> ----
        if (busy) {
            const float4 y0 = *reinterpret_cast<const float4*>(sm.y + c * 8), y1 = *reinterpret_cast<const float4*>(sm.y + c * 8 + 4);
            const float yq[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                float uf[8];
                unpack8_mixed(row(r), uf);
                vals[r] = chunk_partial(yq, uf);
            }
            g_own = reduce_scatter16(vals, c) - s_own;
        }
        if (it == 0) lse = m + logf(Z);
        if (it >= iters) break;
        l_own = have ? ((l_own - m) - eta * g_own) * shrink : -INFINITY;
    }
    // ---- certificate and objective at the final weights a_i = a_own / Z ----
    const float alpha = a_own / Z;
    float sum_ag = have ? alpha * g_own : 0.0f;
    float ent = (have && alpha > 0.0f) ? alpha * ((l_own - m) - logf(Z)) : 0.0f;
    float r2 = 0.0f;
    {
        float qf[8];
        unpack8(q, qf);
#pragma unroll
        for (int e = 0; e < 8; ++e) r2 += (sm.y[c * 8 + e] - qf[e]) * (sm.y[c * 8 + e] - qf[e]);
    }
#pragma unroll
    for (int off = 8; off; off >>= 1) r2 += __shfl_xor_sync(kFullMask, r2, off);
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        sum_ag += __shfl_xor_sync(kFullMask, sum_ag, off);
        ent += __shfl_xor_sync(kFullMask, ent, off);
    }
    // (-g) as a key: the largest key is the smallest gradient entry
    const uint32_t wmin = __reduce_max_sync(kFullMask, have ? float_to_key(-g_own) : 0u);
    if (lane == 0) {
        sm.stat[32 + warp] = wmin;
        stat_f[40 + warp] = sum_ag;
        stat_f[48 + warp] = ent;
    }
    __syncthreads();
    if (tid == 0) {
        uint32_t gk = 0u;
        float sag = 0.0f, en = 0.0f;
        for (int w = 0; w < WARPS; ++w) {
            gk = max(gk, sm.stat[32 + w]);
            sag += stat_f[40 + w];
            en += stat_f[48 + w];
        }
        vsa_solve_t sv;
        sv.fw_gap = sag + key_to_float(gk);   // <g, a> - min_j g_j
        sv.objective = 0.5f * r2 + epsilon * en;
        sv.residual2 = r2;
        sv.step = eta;
        *solve = sv;
    }
    return a_own;
}

// Frank-Wolfe with exact line search on f(a) = 1/2 |sum a_i k_i - q|^2 (App. E).  Vertex choices are integers, so
// everything that feeds them is single-rounded fp32 in the canonical order: the readout y is kept incrementally (lane
// c of a half-warp holds elements 8c .. 8c + 7, every half-warp the same copy), g_i = <k_i, y> - s_i by the fixed-order
// dot, argmin with ties to the lower position, gamma by an IEEE division.  Returns this candidate's weight.
__device__ __forceinline__ float solve_frank_wolfe(const SolveSmem& sm, int ns, float s_own, int pos_own, int iters,
                                                   const uint4& q, vsa_solve_t* solve)
{
    constexpr int WARPS = 8;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c = lane & 15, gi = lane >> 4;
    const bool have = tid < ns, busy = warp * 32 < ns;
    float qf[8];
    unpack8(q, qf);
    // block-wide best (largest key, then lowest position); positions are at most 2^20 and carry the candidate's index;
    // `slot` alternates so that a fast warp cannot overwrite statistics that a slow one still reads
    const uint32_t tag = have ? ((uint32_t)pos_own << 8) | (uint32_t)tid : 0xffffffffu;
    auto arg_best = [&](uint32_t key, int slot, uint32_t& best_key, int& best_j) {
        const uint32_t wk = __reduce_max_sync(kFullMask, key);
        const uint32_t wt = __reduce_min_sync(kFullMask, (key == wk && key != 0u) ? tag : 0xffffffffu);
        if (lane == 0) {
            sm.stat[slot * 16 + warp] = wk;
            sm.stat[slot * 16 + 8 + warp] = wt;
        }
        __syncthreads();
        best_key = 0u;
        uint32_t best_tag = 0xffffffffu;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            const uint32_t k = sm.stat[slot * 16 + w], t = sm.stat[slot * 16 + 8 + w];
            if (k > best_key || (k == best_key && t < best_tag)) {
                best_key = k;
                best_tag = t;
            }
        }
        best_j = (int)(best_tag & 255u);
    };
    auto row_of = [&](int j, float (&x)[8]) { unpack8(*reinterpret_cast<const uint4*>(sm.tile + tile_at(j, c)), x); };
    auto tree16 = [&](float v) {   // canonical halving tree over the half-warp, result in every lane
#pragma unroll
        for (int off = 8; off; off >>= 1) v = v + __shfl_xor_sync(kFullMask, v, off);
        return v;
    };
    uint32_t bk;
    int jb;
    arg_best(have ? float_to_key(s_own) : 0u, 0, bk, jb);
    float yv[8];
    row_of(jb, yv);
    float a_own = (have && tid == jb) ? 1.0f : 0.0f, gamma = 0.0f, gmin = 0.0f;
#pragma unroll 1
    for (int it = 0;; ++it) {
        float g_own = 0.0f;
        if (busy) {
            float vals[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                float uf[8];
                row_of(warp * 32 + gi * 16 + r, uf);
                vals[r] = chunk_partial(yv, uf);
            }
            g_own = reduce_scatter16(vals, c) - s_own;
        }
        // (a NaN gradient, negated, has key 0: as 1 it is the last choice, but one that names a candidate)
        arg_best(have ? max(float_to_key(-g_own), 1u) : 0u, 1 + (it & 1), bk, jb);
        gmin = -key_to_float(bk);
        if (it >= iters) break;
        float uj[8], dv[8], rv[8];
        row_of(jb, uj);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            dv[e] = __fsub_rn(uj[e], yv[e]);
            rv[e] = __fsub_rn(qf[e], yv[e]);
        }
        const float num = tree16(chunk_partial(rv, dv)), den = tree16(chunk_partial(dv, dv));
        gamma = den > 0.0f ? __fdiv_rn(num, den) : 0.0f;
        gamma = gamma < 0.0f ? 0.0f : (gamma > 1.0f ? 1.0f : gamma);
#pragma unroll
        for (int e = 0; e < 8; ++e) yv[e] = __fmaf_rn(gamma, dv[e], yv[e]);
        a_own = __fmaf_rn(-gamma, a_own, a_own);
        if (have && tid == jb) a_own = __fadd_rn(a_own, gamma);
    }
    float rv[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) rv[e] = __fsub_rn(yv[e], qf[e]);
    const float r2 = tree16(chunk_partial(rv, rv)), yr = tree16(chunk_partial(yv, rv));
    if (tid == 0) {
        vsa_solve_t sv;
        sv.fw_gap = __fsub_rn(yr, gmin);
        sv.objective = __fmul_rn(0.5f, r2);
        sv.residual2 = r2;
        sv.step = gamma;
        *solve = sv;
    }
    return a_own;
}

}  // namespace

}  // namespace vsa
