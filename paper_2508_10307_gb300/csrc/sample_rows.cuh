// Sample of the rows of coefficients that an image's groups keep.
#pragma once
#include "kernels.h"

namespace htsvd {

constexpr float G_S3H = 0.866025403784438646763723170752936183f;   // sqrt(3)/2
constexpr float G_SQ3 = 1.73205080756887729352744634150587237f;    // sqrt(3)
constexpr float G_THIRD = 0.333333333333333333333333333333333333f;

// Trailing zeros of 1 <= x < 32 (an expression that folds in unrolled loops; a recursion stays a call there).
__host__ __device__ constexpr int g_ctz(int x) {
    return (x & 1) ? 0 : (x & 2) ? 1 : (x & 4) ? 2 : (x & 8) ? 3 : 4;
}
// sqrt(2^e), the FP32 value (a literal: the square root of a constant is not folded in unrolled loops).
__host__ __device__ constexpr float g_root(int e) {
    return (e & 1) ? 1.41421356237309504880f * (float)(1 << (e >> 1)) : (float)(1 << (e >> 1));
}

// Rows of coefficients that the groups keep, from SR_GROUPS groups spread over the image: one CTA per group
// projects its patches, takes the Haar transform of every coefficient across them and counts the (slot, basis
// row) pairs with a coefficient above the threshold. The last CTA compares the mean with the rows up to which
// the group filter is the faster one (group_rows_limit). 15 us, most of it the latency of one group: the forward pass
// waits for it (a dense image then has no planes), in the backward pass the first blocks of the planes do it.
constexpr int SR_GROUPS = 128;

// Group blk of the sample, by a block of T threads; sm: K patches, [k][i][b or j][NC].
template <int K, int C, typename Tin, bool MF, int T>
__device__ __forceinline__ void sample_group(const FilterArgs& a, int blk, float* sm, unsigned* mask,
                                             int* __restrict__ st, int most) {
    constexpr int NC = C == 3 ? 3 : 1, NF = PS2 * NC;              // floats of a patch
    const Geo& g = a.g;
    const int tid = threadIdx.x, ng = g.nry * g.nrx;
    const int grp = (int)((2ll * blk + 1) * ng / (2 * SR_GROUPS));
    if (tid < PS) mask[tid] = 0u;
#pragma unroll 1
    for (int u = tid; u < K * PS; u += T) {
        // column b of patch k: Y[i][b] = sum_a conj(U[a][i]) X(a, b)
        const int k = u >> 3, b = u & 7;
        int v = max(a.idx[(size_t)grp * K + k], 0);
        const Tin* img = reinterpret_cast<const Tin*>(a.img);
        if constexpr (MF) {
            const int hw = g.H * g.W, f = v / hw;
            img = reinterpret_cast<const Tin*>(a.vid) + (size_t)min(f, a.f0 + a.nfr - 1) * a.fstride;
            v -= f * hw;
        }
        const int y = min(v / g.W, g.H - PS), x = min(v % g.W, g.W - PS);
        float s0[PS] = {}, sr[PS] = {}, si[PS] = {};
#pragma unroll 2
        for (int r = 0; r < PS; ++r) {
            const Tin* p = img + ((size_t)(y + r) * g.W + x + b) * C;
            if constexpr (C == 3) {
                const float v0 = (float)p[0], v1 = (float)p[1], v2 = (float)p[2];
                const float X0 = v0 + v1 + v2, Xr = v0 - 0.5f * (v1 + v2), Xi = G_S3H * (v2 - v1);
#pragma unroll
                for (int i = 0; i < PS; ++i) {
                    const float ur = a.basis32[64 + r * PS + i], ui = a.basis32[128 + r * PS + i];
                    s0[i] = fmaf(a.basis32[r * PS + i], X0, s0[i]);
                    sr[i] = fmaf(ur, Xr, fmaf(ui, Xi, sr[i]));
                    si[i] = fmaf(ur, Xi, fmaf(-ui, Xr, si[i]));
                }
            } else {
                const float X0 = (float)p[0];
#pragma unroll
                for (int i = 0; i < PS; ++i) s0[i] = fmaf(a.basis32[r * PS + i], X0, s0[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < PS; ++i) {
            float* d = sm + k * NF + (i * PS + b) * NC;
            d[0] = s0[i];
            if constexpr (C == 3) {
                d[1] = sr[i];
                d[2] = si[i];
            }
        }
    }
    __syncthreads();
#pragma unroll 1
    for (int u = tid; u < K * PS; u += T) {
        // row i of patch k: S[i][j] = sum_b Y[i][b] V[b][j] and the inverse channel DFT, over its own floats
        float* row = sm + (u >> 3) * NF + (u & 7) * PS * NC;
        float s0[PS] = {}, sr[PS] = {}, si[PS] = {};
        const float* V = a.basis32 + (C == 3 ? 192 : 64);
#pragma unroll 2
        for (int b = 0; b < PS; ++b) {
            const float y0 = row[b * NC], yr = C == 3 ? row[b * NC + (C == 3 ? 1 : 0)] : 0.f;
            const float yi = C == 3 ? row[b * NC + (C == 3 ? 2 : 0)] : 0.f;
#pragma unroll
            for (int j = 0; j < PS; ++j) {
                s0[j] = fmaf(y0, V[b * PS + j], s0[j]);
                if constexpr (C == 3) {
                    const float vr = V[64 + b * PS + j], vi = V[128 + b * PS + j];
                    sr[j] = fmaf(yr, vr, fmaf(-yi, vi, sr[j]));
                    si[j] = fmaf(yr, vi, fmaf(yi, vr, si[j]));
                }
            }
        }
#pragma unroll
        for (int j = 0; j < PS; ++j) {
            if constexpr (C == 3) {
                row[j * 3] = (s0[j] + 2.f * sr[j]) * G_THIRD;
                row[j * 3 + 1] = (s0[j] - sr[j] - G_SQ3 * si[j]) * G_THIRD;
                row[j * 3 + 2] = (s0[j] - sr[j] + G_SQ3 * si[j]) * G_THIRD;
            } else {
                row[j] = s0[j];
            }
        }
    }
    __syncthreads();
    for (int t = tid; t < NF; t += T) {
        // coefficient t across the patches (unnormalised: the threshold grows with the support)
        float p[K];
#pragma unroll
        for (int k = 0; k < K; ++k) p[k] = sm[k * NF + t];
#pragma unroll
        for (int d = 1; d < K; d <<= 1)
#pragma unroll
            for (int m = 0; m < K; m += 2 * d) {
                const float x = p[m], y = p[m + d];
                p[m + d] = x - y;
                p[m] = x + y;
            }
        unsigned keep = 0u;
#pragma unroll
        for (int l = 0; l < K; ++l)
            if (fabsf(p[l]) >= a.tau32 * g_root(l == 0 ? g_ctz(K) : g_ctz(l) + 1)) keep |= 1u << l;
        atomicOr(&mask[t / (PS * NC)], keep);
    }
    __syncthreads();
    if (tid == 0) {
        int rows = 0;
        for (int i = 0; i < PS; ++i) rows += __popc(mask[i]);
        atomicAdd(st, rows);
        __threadfence();
        if (atomicAdd(st + 1, 1) == SR_GROUPS - 1) st[2] = atomicAdd(st, 0) > most;
    }
}

}  // namespace htsvd
