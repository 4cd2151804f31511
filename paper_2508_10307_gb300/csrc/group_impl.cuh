// Group filter on projection planes (Alg. 1 Steps 2(2)-(4) and 3 after the patches' projection).
//
// Every group is one warp's work from end to end, so no CTA barrier paces it; the warps of a CTA share a tile
// of references and its footprint accumulator and take the tile's groups in turn:
//   1  gather: lane (i, j) of half h reads the C channels of coefficient (4 h + i, j) of the K patches
//      from the projection planes (coalesced), all K patches in flight;
//   2  Haar analysis in registers, two values per packed operation; slots where no lane can keep a
//      coefficient are ruled out by one comparison each, the others thresholded one by one (FP64 decision
//      inside the guard band). A slot leaves the basis rows that kept a coefficient, after the channel
//      DFT, in a compacted list in shared memory;
//   3  Z_f[i, :] = T_f[i, :] V_f^H for the listed rows, four rows at a time (lane = row, column b);
//   4  depth-first over the Haar synthesis tree: at a node, U_f Z_f over the slot's listed rows and the
//      inverse channel DFT for the lane's two pixels (a, 2 b2), (a, 2 b2 + 1) as packed pairs, then
//      sum and difference to the two children; a leaf is an estimated patch and is added to the
//      footprint at once. The warps hand the accumulator over in group order (named barriers), so
//      the sums have a fixed order: bitwise reproducible.
// The sums at each step have the term order of filter_tile_fwd, so both give the same partials.
// Rows beyond the list's shared-memory capacity go to a per-warp spill buffer in global memory.
//
// Bound by instruction issue and by the serial chain of a group (issue slots 39 % busy): a group keeps
// coefficients in some 20 of its 256 (slot, basis row) pairs at the default threshold, so the inverse is a small
// part of the dense one, and what is left is the gather, the analysis and K leaves. Three warps a CTA: 9.7 ms for a
// 3840 x 2160 RGB frame at K 32, window 31 (2 warps: 12.5, 4: 12.0; four listed rows per step of the inverse:
// 13.5, the loop outgrows the instruction cache). The projection in the CTA and dense inverse of filter_tile_fwd
// took 20.3 ms; with the planes (1.3 ms) this is 11.0. 1920 x 1080 gray: 2.56 -> 1.56 + 0.09 ms.
#pragma once
#include "f32x2.cuh"
#include <type_traits>

#include "kernels.h"
#include "sample_rows.cuh"

namespace htsvd {

constexpr int GR_WARPS = 3;                  // warps per CTA (and tile)
constexpr int GR_THREADS = GR_WARPS * 32;
constexpr int GR_CTAS = 16 / GR_WARPS;       // CTAs per SM that the registers allow (16 warps of 128 registers)
constexpr int GR_RAW = 4;                    // slots' raw coefficients that fit behind a full row list
template <int C>
struct GCfg {
    static constexpr int ACC = (C == 3) ? 4 : 2;      // floats per footprint pixel
    static constexpr int RW = PS * C;                 // floats per listed row
    static constexpr int UF = (C == 3) ? 8 : 2;       // floats per (i, a) of the U table (duplicated pairs)
};

// Shared memory (bytes): U and V tables, per-warp tables, accumulator, per-warp row lists.
struct GLayout {
    int off_u, off_v, off_tab, off_acc, off_list, total;
};
template <int C>
__host__ __device__ inline GLayout group_layout(int FHmax, int FWmax, int cap, bool adj) {
    GLayout L;
    int o = 0;
    L.off_u = o; o += PS2 * GCfg<C>::UF * 4;
    L.off_v = o; o += (C == 3 ? 3 : 1) * PS2 * 4;
    L.off_tab = o; o += GR_WARPS * 32 * 4;             // per warp: 32 position words
    L.off_acc = o; o += FHmax * (FWmax | 1) * GCfg<C>::ACC * 4;
    o = (o + 15) & ~15;                                // (cleared in 16-byte words)
    L.off_list = o; o += GR_WARPS * (cap * GCfg<C>::RW + GR_RAW * (C == 3 ? 96 : 64) * (adj ? 2 : 1)) * 4;
    L.total = o;
    return L;
}

// Loads of one patch's coefficients, kept in program order (ahead of their use, one address at a time).
__device__ __forceinline__ f2 ldg_pair(const float* p) {
    f2 v;
    asm volatile("ld.global.nc.b64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ldg_one(const float* p) {
    float v;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// A pair of a constant that stays in registers (not rebuilt at each use).
__device__ __forceinline__ f2 f2_held(float x) {
    f2 r;
    asm volatile("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// If bit is set in mask: the pair (and the single value, d1 bytes on) to shared address d, which moves on by
// STEP bytes. Predicated stores, no branch.
template <int NS, int STEP>
__device__ __forceinline__ void stage_slot(uint32_t mask, const uint32_t bit, uint32_t& d, uint32_t d1, f2 pair, float one) {
    if constexpr (NS) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.b32 p, t, 0;\n\t"
            "@p st.shared.b64 [%0], %3;\n\tadd.u32 t, %0, %4;\n\t@p st.shared.f32 [t], %5;\n\t@p add.u32 %0, %0, %6;\n\t}"
            : "+r"(d)
            : "r"(mask), "r"(bit), "l"(pair), "r"(d1), "f"(one), "n"(STEP)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.b32 p, t, 0;\n\t"
            "@p st.shared.b64 [%0], %3;\n\t@p add.u32 %0, %0, %4;\n\t}"
            : "+r"(d)
            : "r"(mask), "r"(bit), "l"(pair), "n"(STEP)
            : "memory");
    }
}

__host__ __device__ constexpr int g_log2(int k) { return k <= 1 ? 0 : 1 + g_log2(k / 2); }
// Floats of global scratch per warp.
__host__ __device__ constexpr size_t group_spill_warp(int K, int C) {
    return (size_t)K * PS * PS * C + (size_t)2 * K * (4 + 3 * 32);
}

// FP64 value of coefficient (Haar row m, fibre e) of the group against tau64, by the whole warp: lane l
// takes the pixels l and l + 32 of the combined patch. lin: lane k's patch position (linear pixel index
// into img); for uint8 inputs the signed sum of the patches is exact in int32.
template <int C, typename Tin>
__device__ __noinline__ bool group_refine(int m, int e, int K, const Tin* __restrict__ img, int W, int lin,
                                          const double* __restrict__ b64, double tau64, int lane) {
    int k0 = 0, L = K;
    if (m > 0) {
        const int l = 31 - __clz(m);
        L = K >> l;
        k0 = (m - (1 << l)) * L;
    }
    const int half = (m == 0) ? L : L / 2;
    const int e2 = 31 - __clz(L);
    const double hh = ldexp((e2 & 1) ? 0.70710678118654752440 : 1.0, -(e2 >> 1));
    const int pix = e / C, ch = e - pix * C;
    const int i = pix / PS, j = pix % PS;
    const double s3h = 0.5 * sqrt(3.0);
    double s0 = 0.0, s1r = 0.0, s1i = 0.0;
#pragma unroll 1
    for (int rep = 0; rep < 2; ++rep) {
        const int p = lane + 32 * rep;
        const int aa = p / PS, bb = p % PS;
        double q[C];
        int qi[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            q[c] = 0.0;
            qi[c] = 0;
        }
        for (int kk = k0; kk < k0 + L; ++kk) {
            const long long base = (long long)__shfl_sync(0xffffffffu, lin, kk) + (long long)aa * W + bb;
            const bool pos = kk - k0 < half;
#pragma unroll
            for (int c = 0; c < C; ++c) {
                if constexpr (sizeof(Tin) == 1) {
                    const int v = (int)img[base * C + c];
                    qi[c] += pos ? v : -v;
                } else {
                    const double v = (double)img[base * C + c];
                    q[c] += pos ? v : -v;
                }
            }
        }
#pragma unroll
        for (int c = 0; c < C; ++c) q[c] = (sizeof(Tin) == 1 ? (double)qi[c] : q[c]) * hh;
        const double u0 = b64[2 * (aa * PS + i)];
        const double v0 = b64[C * 2 * PS2 + 2 * (bb * PS + j)];
        if constexpr (C == 3) {
            const double Q0 = q[0] + q[1] + q[2];
            const double Q1r = q[0] - 0.5 * (q[1] + q[2]);
            const double Q1i = s3h * (q[2] - q[1]);
            s0 += u0 * Q0 * v0;
            const double u1r = b64[2 * PS2 + 2 * (aa * PS + i)];
            const double u1i = b64[2 * PS2 + 2 * (aa * PS + i) + 1];
            const double v1r = b64[(C + 1) * 2 * PS2 + 2 * (bb * PS + j)];
            const double v1i = b64[(C + 1) * 2 * PS2 + 2 * (bb * PS + j) + 1];
            const double tr = u1r * Q1r + u1i * Q1i;       // conj(u1) * Q1
            const double ti = u1r * Q1i - u1i * Q1r;
            s1r += tr * v1r - ti * v1i;
            s1i += tr * v1i + ti * v1r;
        } else {
            s0 += u0 * q[0] * v0;
        }
    }
    double S = s0;
    if constexpr (C == 3) {
        const double sq3 = sqrt(3.0), third = 1.0 / 3.0;
        S = (ch == 0) ? (s0 + 2.0 * s1r) * third : (ch == 1) ? (s0 - s1r - sq3 * s1i) * third
                                                              : (s0 - s1r + sq3 * s1i) * third;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) S += __shfl_xor_sync(0xffffffffu, S, off);
    return fabs(S) >= tau64;
}

// Guard-band record of one Haar slot (global scratch): the slot and half, per value of a lane the lanes
// whose coefficient lies inside the group-wide band (rewritten with the lanes that keep it), and the
// distances of the coefficients to the threshold.
struct BandRec {
    uint32_t head, lanes[3];
    float d[3][32];
};

// Decides the recorded coefficients of one group. The FP32 error of a slot's row only involves the
// patches of its support, so the band first narrows to their norm; what stays inside is recomputed in
// FP64 by the whole warp. pnk, lin: lane k's patch norm and position.
template <int C, typename Tin>
__device__ __noinline__ void group_band(const FilterArgs& a, BandRec* rec, int n, float pnk, int lin, int lane) {
    const int K = a.g.K;
    const Tin* img = reinterpret_cast<const Tin*>(a.mode == FM_VIDEO ? a.vid : a.img);
    for (int r = 0; r < n; ++r) {
        const uint32_t head = rec[r].head;
        const int sl = head & 255u, h = head >> 8;
        const int L = sl == 0 ? K : 2 << (__ffs(sl) - 1);
        const int m = sl == 0 ? 0 : K / L + sl / L;
        const int k0 = sl == 0 ? 0 : (sl / L) * L;
        float sq = (lane >= k0 && lane < k0 + L) ? pnk : 0.f;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
        const float lim = (a.band_rel * sqrtf(sq) + a.band_abs) * sqrtf((float)L);
        for (int v = 0; v < (C == 3 ? 3 : 2); ++v) {
            const uint32_t in = rec[r].lanes[v];
            const float d = rec[r].d[v][lane];
            const bool mine = (in >> lane) & 1u;
            uint32_t keep = __ballot_sync(0xffffffffu, mine && fabsf(d) > lim && d >= 0.f);
            uint32_t open = __ballot_sync(0xffffffffu, mine && !(fabsf(d) > lim));
            while (open) {
                const int l = __ffs(open) - 1;
                open &= open - 1;
                const int hh = C == 3 ? h : v;
                const int e = ((4 * hh + (l >> 3)) * PS + (l & 7)) * C + (C == 3 ? v : 0);
                if (group_refine<C, Tin>(m, e, K, img, a.g.W, lin, a.basis64, a.tau64, lane)) keep |= 1u << l;
            }
            if (lane == 0) rec[r].lanes[v] = keep;
        }
    }
    __syncwarp();
}

// The inverse of one group from its row list: values of the Haar slots, synthesis, aggregation.
template <int K, int C, bool MF, bool SP>
struct Inverse {
    using G = GCfg<C>;
    static constexpr int LV = g_log2(K);
    uint32_t slots;          // lane sl, per slot: half 0 in the low 16 bits, half 1 in the high: row mask | first row << 4
    const float* list;       // + 2 pb
    const float* spill;
    int cap;
    const float* ub;         // U table + pa
    float* acc;              // + this lane's pixel offset
    int aoff;                // lane k: accumulator offset of patch k (-1: not aggregated)
    float wg;
    f2 third, sq3, nsq3;     // constants of the inverse channel DFT, held in registers

    // dv = the slot's values at this lane's two pixels (zero if the slot kept nothing).
    __device__ __forceinline__ void value(int sl, f2 (&dv)[C]) const {
        const uint32_t word = __shfl_sync(0xffffffffu, slots, sl);
#pragma unroll
        for (int c = 0; c < C; ++c) dv[c] = 0;
        if (word == 0u) return;                        // warp-uniform
        f2 g0 = 0, gr = 0, gi = 0;
        uint32_t rest = word;                          // half 0, then half 1 (rows 4 .. 7)
        const float* u0 = ub;
        // (rolled: taking four or two rows at a time, their loads first, made the loop outgrow the instruction
        // cache: 9.7 -> 13.5 ms per 3840 x 2160 frame)
#pragma unroll 1
        do {
            int rr = (rest >> 4) & 0xfffu;
            const float* z = list + rr * G::RW;
#pragma unroll 1
            for (uint32_t m = rest & 15u; m; m &= m - 1, z += G::RW, ++rr) {
                const float* u = u0 + (__ffs(m) - 1) * PS * G::UF;
                f2 z0, zr, zi;
                if (SP && rr >= cap) {
                    const float* q = spill + (rr - cap) * G::RW;
                    z0 = *reinterpret_cast<const f2*>(q);
                    if constexpr (C == 3) {
                        zr = *reinterpret_cast<const f2*>(q + 8);
                        zi = *reinterpret_cast<const f2*>(q + 16);
                    }
                } else {
                    z0 = *reinterpret_cast<const f2*>(z);
                    if constexpr (C == 3) {
                        zr = *reinterpret_cast<const f2*>(z + 8);
                        zi = *reinterpret_cast<const f2*>(z + 16);
                    }
                }
                if constexpr (C == 3) {
                    const ulonglong2 u01 = *reinterpret_cast<const ulonglong2*>(u);
                    const ulonglong2 u23 = *reinterpret_cast<const ulonglong2*>(u + 4);
                    g0 = f2_fma(u01.x, z0, g0);
                    gr = f2_fma(u01.y, zr, f2_fma(u23.y, zi, gr));
                    gi = f2_fma(u01.y, zi, f2_fma(u23.x, zr, gi));
                } else {
                    g0 = f2_fma(*reinterpret_cast<const f2*>(u), z0, g0);
                }
            }
            rest >>= 16;
            u0 += 4 * PS * G::UF;
        } while (rest);
        if constexpr (C == 3) {
            const f2 d01 = f2_sub(g0, gr);
            dv[0] = f2_mul(f2_add(f2_add(gr, gr), g0), third);     // (2 gr is exact)
            dv[1] = f2_mul(f2_fma(nsq3, gi, d01), third);
            dv[2] = f2_mul(f2_fma(sq3, gi, d01), third);
        } else {
            dv[0] = g0;
        }
    }
    // Adds the estimated patch k.
    __device__ __forceinline__ void leaf(int k, const f2 (&val)[C]) const {
        const int off = __shfl_sync(0xffffffffu, aoff, k);
        if (MF && off < 0) return;                     // a patch of another frame
        float* d = acc + off;
        float x0[C], x1[C];
#pragma unroll
        for (int c = 0; c < C; ++c) f2_unpack(val[c], x0[c], x1[c]);
        if constexpr (C == 3) {
            float4 t0 = reinterpret_cast<float4*>(d)[0], t1 = reinterpret_cast<float4*>(d)[1];
            t0.x = fmaf(wg, x0[0], t0.x); t1.x = fmaf(wg, x1[0], t1.x);
            t0.y = fmaf(wg, x0[1], t0.y); t1.y = fmaf(wg, x1[1], t1.y);
            t0.z = fmaf(wg, x0[2], t0.z); t1.z = fmaf(wg, x1[2], t1.z);
            t0.w += wg; t1.w += wg;
            reinterpret_cast<float4*>(d)[0] = t0;
            reinterpret_cast<float4*>(d)[1] = t1;
        } else {
            float2 t0 = reinterpret_cast<float2*>(d)[0], t1 = reinterpret_cast<float2*>(d)[1];
            t0.x = fmaf(wg, x0[0], t0.x); t1.x = fmaf(wg, x1[0], t1.x);
            t0.y += wg; t1.y += wg;
            reinterpret_cast<float2*>(d)[0] = t0;
            reinterpret_cast<float2*>(d)[1] = t1;
        }
        __syncwarp();                                  // orders the updates of patches k, k + 1
    }
    // Node idx of level l with value v: its slot's value to the two children, the left subtree first.
    template <int l>
    __device__ __forceinline__ void node(int idx, const f2 (&v)[C]) const {
        if constexpr (l == LV) {
            leaf(idx, v);
        } else {
            f2 d[C], x[C];
            value((2 * idx + 1) * (K >> (l + 1)), d);
#pragma unroll
            for (int c = 0; c < C; ++c) x[c] = f2_add(v[c], d[c]);
            node<l + 1>(2 * idx, x);
#pragma unroll
            for (int c = 0; c < C; ++c) x[c] = f2_sub(v[c], d[c]);
            node<l + 1>(2 * idx + 1, x);
        }
    }
    // The whole tree: subtrees of at most 4 leaves unrolled (the instruction cache holds the kernel's loop),
    // the levels above in a loop over them: level i's value is formed when its node begins, and the path's
    // sums are taken again for each subtree.
    __device__ __forceinline__ void run() const {
        constexpr int TL = LV > 2 ? LV - 2 : 0;
        f2 root[C], d[TL > 0 ? TL : 1][C];
        value(0, root);
#pragma unroll 1
        for (int t = 0; t < (1 << TL); ++t) {
            f2 v[C];
#pragma unroll
            for (int c = 0; c < C; ++c) v[c] = root[c];
#pragma unroll
            for (int i = 0; i < TL; ++i) {
                if ((t & ((1 << (TL - i)) - 1)) == 0) value((2 * (t >> (TL - i)) + 1) * (K >> (i + 1)), d[i]);
                const f2 sg = f2_dup(((t >> (TL - 1 - i)) & 1) ? -1.f : 1.f);
#pragma unroll
                for (int c = 0; c < C; ++c) v[c] = f2_fma(sg, d[i][c], v[c]);
            }
            node<TL>(t, v);
        }
    }
};

// One gather step: the coefficients of KB = K/2 patches (planes at src, positions pos), then their Haar
// analysis (unnormalised, in place). C = 3: p holds channels 0 and 1, s channel 2; C = 1: p holds both halves.
template <int K, int C>
__device__ __forceinline__ void gather_haar(const float* src, const uint32_t* pos, int lane, f2 (&p)[K / 2],
                                            float (&s)[C == 3 ? K / 2 : 1]) {
    constexpr int KB = K / 2, NS = C == 3 ? 1 : 0, NF = PS2 * C;
    if constexpr (KB >= 4) {
#pragma unroll
        for (int k = 0; k < KB; k += 4) {
            const uint4 o = *reinterpret_cast<const uint4*>(pos + k);
            const uint32_t oo[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const float* t = src + (size_t)oo[u] * NF;
                p[k + u] = ldg_pair(t);
                if constexpr (NS) s[k + u] = ldg_one(t + 64 - lane);
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < KB; ++k) {
            const float* t = src + (size_t)pos[k] * NF;
            p[k] = ldg_pair(t);
            if constexpr (NS) s[k] = ldg_one(t + 64 - lane);
        }
    }
#pragma unroll
    for (int d = 1; d < KB; d <<= 1)
#pragma unroll
        for (int m = 0; m < KB; m += 2 * d) {
            const f2 x = p[m], y = p[m + d];
            p[m + d] = f2_sub(x, y);
            p[m] = f2_add(x, y);
            if constexpr (NS) {
                const float u = s[m], v = s[m + d];
                s[m + d] = u - v;
                s[m] = u + v;
            }
        }
}

// MF: patches of several frames. ADJ: the transposed map at the image (masks from its planes, the
// coefficients that are inverted from the planes of r = gout / D), with the gradient of the group weights
// <kept coefficients of r, of the image> - <patches of r, patches of the output>.
template <int K, int C, typename Tin, bool MF, bool ADJ>
__device__ __forceinline__ void group_tile(const GroupArgs& A, const int ty, const int tx, unsigned char* smem,
                                           float* __restrict__ spill, int* probe) {
    using G = GCfg<C>;
    constexpr int NF = PS2 * C;
    constexpr int NBW = K * NF / 32;
    constexpr int LV = g_log2(K);
    constexpr int NS = C == 3 ? 1 : 0;                 // unpaired values per lane (channel 2)
    constexpr int NH = C == 3 ? 1 : 2;                 // halves per gather pass
    constexpr int NV = 2 + NS;                         // values per lane and slot
    constexpr int ONE = 64 + 32 * NS;                  // staged words per slot and image
    constexpr int RAWF = ADJ ? 2 * ONE : ONE;
    constexpr int KB = K / 2;                          // patches per gather step
    constexpr unsigned FULL = 0xffffffffu;
    const FilterArgs& a = A.f;
    const Geo& g = a.g;
    // (the warp index by a shuffle: the compiler then knows it, and the control flow it drives, as uniform)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    int FY0, FY1, FX0, FX1;
    tile_span(ty, a.TR, g.nry, g.s, g.H, g.npy, g.wny, g.win, FY0, FY1);
    tile_span(tx, a.TR, g.nrx, g.s, g.W, g.npx, g.wnx, g.win, FX0, FX1);
    const int FH = FY1 - FY0, FW = FX1 - FX0;
    const int FWp = a.FWmax | 1;                       // odd pitch: a quarter warp's two pixel rows fall on
                                                       // different bank groups
    const GLayout L = group_layout<C>(a.FHmax, a.FWmax, A.cap, ADJ);
    const float* ut = reinterpret_cast<const float*>(smem + L.off_u);
    const float* vt = reinterpret_cast<const float*>(smem + L.off_v);
    uint32_t* posw = reinterpret_cast<uint32_t*>(smem + L.off_tab) + warp * 32;
    float* acc = reinterpret_cast<float*>(smem + L.off_acc);
    float* list = reinterpret_cast<float*>(smem + L.off_list) + warp * (A.cap * G::RW + GR_RAW * RAWF);
    // per-warp global scratch: spilled rows, then the guard-band records (one per slot and half at most)
    spill += (size_t)warp * group_spill_warp(K, C);
    BandRec* rec = reinterpret_cast<BandRec*>(spill + K * PS * G::RW);
    const int cap = A.cap;

    for (int t = tid; t < (FH * FWp * G::ACC + 3) / 4; t += GR_THREADS)
        reinterpret_cast<float4*>(acc)[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int iy0 = ty * a.TR, ix0 = tx * a.TR;
    const int th = min(a.TR, g.nry - iy0), tw = min(a.TR, g.nrx - ix0);
    const int ngr = th * tw;
    auto group_of = [&](int q) { return (iy0 + q / tw) * g.nrx + ix0 + q % tw; };
    int grp = warp < ngr ? group_of(warp) : 0;         // group of this warp's turn
    int qx = warp % tw;

    const int b = lane & 7;                            // row column of stage D
    const unsigned rowbit = 0x80u << (lane & 24);      // this lane's basis row in the row mask, and the rows below
    const unsigned below = (1u << (lane & 24)) - 1u;
    // pixels of stage E: (pa, 2 pb), (pa, 2 pb + 1)
    const int pa = lane >> 2, pb = lane & 3;
    const int lane_off = (pa * FWp + 2 * pb) * G::ACC;
    const f2 third = f2_held(G_THIRD), sq3 = f2_held(G_SQ3), nsq3 = f2_held(-G_SQ3);
    float rtab = 1.f;                                  // lane e: sqrt(2^e)
#pragma unroll
    for (int e = 1; e < 6; ++e) rtab = lane == e ? g_root(e) : rtab;

    int next = (warp < ngr && lane < K) ? a.idx[(size_t)grp * K + lane] : 0;
    if (tid == 0) *probe = 0;
    __syncthreads();                                   // accumulator cleared, tables staged
    const int first = min(ngr, GR_WARPS);              // groups of the first turns
    if (warp >= ngr) __syncthreads();                  // (no turn: the barrier of the others' first one)
    bool left = false;                                 // (the same in every warp that has a turn)

#pragma unroll 1
    for (int q = warp; q < ngr; q += GR_WARPS) {
        int ahead = grp + GR_WARPS;                    // group of turn q + GR_WARPS
        qx += GR_WARPS;
        while (qx >= tw) {
            qx -= tw;
            ahead += g.nrx - tw;
        }
        // ---- lane k: patch k of the group
        int lin = 0, aoff = 0;
        float pnk = 0.f, dots = 0.f;
        {
            int v = next, f = 0;
            uint32_t ppos = 0;
            if (lane < K) {
                bool mine = true;
                v = max(v, 0);
                if (MF) {                              // clamped to the staged frames
                    const int hw = g.H * g.W;
                    const int vf = v / hw;
                    f = min(max(vf, a.f0), a.f0 + a.nfr - 1);
                    v -= vf * hw;
                    mine = f == a.fref;
                }
                // Positions come from the grouping of this geometry and lie in the footprint; a caller-given
                // index outside it is clamped so that no access leaves the planes or the accumulator.
                int yy = (int)__umulhi((unsigned)v, A.wrec);       // v / W from 2^32 / W rounded down: one short at most
                int xx = v - yy * g.W;
                if (xx >= g.W) {
                    ++yy;
                    xx -= g.W;
                }
                const int fy = min(max(yy - FY0, 0), FH - PS), fx = min(max(xx - FX0, 0), FW - PS);
                lin = f * g.H * g.W + (FY0 + fy) * g.W + FX0 + fx;
                aoff = mine ? (fy * FWp + fx) * G::ACC : -1;
                ppos = (uint32_t)((MF ? (f - a.f0) * A.planestride : 0) + (long long)(FY0 + fy - A.py0) * g.npx + FX0 + fx);
                pnk = A.pn[ppos];
                if constexpr (ADJ) dots = -A.dot[ppos];
            }
            __syncwarp();
            posw[lane] = ppos;
            __syncwarp();
        }
        next = (q + GR_WARPS < ngr && lane < K) ? a.idx[(size_t)ahead * K + lane] : 0;

        float delta = 0.f, lo1 = 0.f;
        int nrow = 0, kept = 0;
        float dot_all = 0.f;
        uint32_t slots = 0;                            // lane sl: kept rows of slot sl (see Inverse)
        // A second pass follows where coefficients lie inside the guard band: the first records them, and
        // the FP64 decisions come in between, when no coefficients are held in registers.
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
        int nrec = 0;
        f2 root = 0, rroot = 0;                        // first half of the group's Haar sum (see below)
        float roots = 0.f, rroots = 0.f, dot = 0.f;
        bool have_r = false;
        nrow = kept = 0;
        slots = 0;
#pragma unroll 1
        for (int st = 0; st < 2 * (2 / NH); ++st) {
            // Step (half h0, patches k0 .. k0 + KB - 1): the Haar details within K/2 patches need no others,
            // so a lane holds K/2 patches at a time, and the two partial sums meet at the end of a half.
            const int h0 = st >> 1, k0 = (st & 1) * KB;
            // ---- gather: C = 3: the channels of coefficient (4 h0 + lane / 8, lane % 8), channels 0 and 1 as
            // one pair; C = 1: both halves' coefficients as one pair
            f2 p[KB];
            float s[NS ? KB : 1];
            gather_haar<K, C>(A.coef + h0 * 32 * C + lane * 2, posw + k0, lane, p, s);
            if (st == 0) {
                float nrm2 = pnk;
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) nrm2 += __shfl_xor_sync(FULL, nrm2, off);
                delta = a.band_rel * sqrtf(nrm2) + a.band_abs;
                lo1 = (a.tau32 - delta) * (1.f - 1e-6f) - 1e-30f;   // below it nothing is kept or in the band
            }
            // the last level: slot 0 (sum) and slot K/2 (difference) once both partial sums are there
            f2 top = 0;
            float tops = 0.f;
            const bool last = k0 != 0;
            if (last) {
                top = f2_sub(root, p[0]);
                p[0] = f2_add(root, p[0]);
                if constexpr (NS) {
                    tops = roots - s[0];
                    s[0] = roots + s[0];
                }
            } else {
                root = p[0];
                if constexpr (NS) roots = s[0];
            }
            // value of local slot l: l < KB in place, l = KB the last level's difference
            auto pair_at = [&](int l) { return l < KB ? p[l < KB ? l : 0] : top; };
            auto one_at = [&](int l) { return l < KB ? s[NS && l < KB ? l : 0] : tops; };
            if (a.coef_out) {
                float* cdst = a.coef_out + (size_t)grp * K * NF;
#pragma unroll
                for (int l = 0; l <= KB; ++l) {
                    if ((l == 0 || l == KB) && !last) continue;
                    const int gs = l == 0 ? 0 : l == KB ? KB : k0 + l;
                    const int e = l == 0 || l == KB ? LV : g_ctz(l) + 1;
                    const float n = 1.f / g_root(e);
                    float* o = cdst + (gs == 0 ? 0 : (K >> e) + (gs >> e)) * NF;
                    if constexpr (C == 3) {
                        o += (h0 * 32 + lane) * 3;
                        o[0] = f2_lo(pair_at(l)) * n;
                        o[1] = f2_hi(pair_at(l)) * n;
                        o[2] = one_at(l) * n;
                    } else {
                        o[lane] = f2_lo(pair_at(l)) * n;
                        o[32 + lane] = f2_hi(pair_at(l)) * n;
                    }
                }
            }
            // ---- local slots where some lane may keep a coefficient
            uint32_t act = 0;
            float lo[LV + 1];
#pragma unroll
            for (int e = 1; e <= LV; ++e) lo[e] = lo1 * g_root(e);
#pragma unroll
            for (int l = 0; l <= KB; ++l) {
                float mx = fmaxf(fabsf(f2_lo(pair_at(l))), fabsf(f2_hi(pair_at(l))));
                if constexpr (NS) mx = fmaxf(mx, fabsf(one_at(l)));
                if (!(mx < lo[l == 0 || l == KB ? LV : g_ctz(l) + 1])) act |= 1u << l;
            }
            if (!last) act &= ~(1u | (1u << KB));
            if (q < GR_WARPS && pass == 0 && st == 0) {
                // A tile most of whose first groups may keep many (slot, basis row) pairs in this step is left
                // to the kernel that works through every row alike (filter_tile_fwd), before any of its
                // coefficients is taken up.
                uint32_t m = act;
                m |= __shfl_xor_sync(FULL, m, 1);
                m |= __shfl_xor_sync(FULL, m, 2);
                m |= __shfl_xor_sync(FULL, m, 4);
                int rows = __popc(m);                  // of the lane's basis row
                rows += __shfl_xor_sync(FULL, rows, 8);
                rows += __shfl_xor_sync(FULL, rows, 16);
                if (lane == 0 && rows > A.dense_rows) atomicAdd(probe, 1);
                __syncthreads();
                if (2 * probe[0] > first) {
                    left = true;
                    break;
                }
            }
            act = __reduce_or_sync(FULL, act);
            f2 q2[ADJ ? KB : 1], rtop = 0;             // ADJ: the same coefficients of r
            float qs[ADJ && NS ? KB : 1], rtops = 0.f;
            if constexpr (ADJ) {
                const float* rsrc = A.rcoef + h0 * 32 * C + lane * 2;
                if (act != 0u || (h0 == 0 && !last)) {     // (half 0 keeps something in almost every group)
                    gather_haar<K, C>(rsrc, posw + k0, lane, q2, qs);
                    if (last) {
                        if (!have_r) {                     // the first partial sum was not needed until now
                            rroot = 0;
                            rroots = 0.f;
#pragma unroll 1
                            for (int k = 0; k < KB; ++k) {
                                const float* t = rsrc + (size_t)posw[k] * NF;
                                rroot = f2_add(rroot, ldg_pair(t));
                                if constexpr (NS) rroots += ldg_one(t + 64 - lane);
                            }
                        }
                        rtop = f2_sub(rroot, q2[0]);
                        q2[0] = f2_add(rroot, q2[0]);
                        if constexpr (NS) {
                            rtops = rroots - qs[0];
                            qs[0] = rroots + qs[0];
                        }
                    } else {
                        rroot = q2[0];
                        if constexpr (NS) rroots = qs[0];
                    }
                    have_r = true;
                } else {
                    have_r = false;
                }
            }
            // ---- threshold, a batch of active slots at a time: their raw coefficients are staged behind the
            // row list (static register indices), then taken up by a rolled loop. A slot's staged words
            // cover the rows it can add, so the list grows over them as they are read.
#pragma unroll 1
            while (act) {
                float* raw = list + min(nrow, cap) * G::RW;
                const int room = max(cap - nrow, 0) * G::RW / RAWF + GR_RAW;
                uint32_t sub = act;
                if (__popc(act) > room) sub = act & ((2u << __fns(act, 0, room)) - 1u);
                act &= ~sub;
                uint32_t d = smem_addr(raw + lane * 2);
                const uint32_t d1 = 256u - 4u * lane;
#pragma unroll
                for (int l = 0; l <= KB; ++l) {
                    if constexpr (ADJ) {
                        uint32_t dr = d + ONE * 4;
                        stage_slot<NS, 0>(sub, 1u << l, dr, d1, l < KB ? q2[ADJ && l < KB ? l : 0] : rtop,
                                          l < KB ? qs[ADJ && NS && l < KB ? l : 0] : rtops);
                    }
                    stage_slot<NS, RAWF * 4>(sub, 1u << l, d, d1, pair_at(l), one_at(l));
                }
                __syncwarp();
                const float* src = raw + lane * 2;
#pragma unroll 1
                for (; sub; sub &= sub - 1, src += RAWF) {
                    const int l = __ffs(sub) - 1;
                    const int e = __ffs(l | KB);                            // support 2^e
                    const float r = __shfl_sync(FULL, rtab, e);
                    const float2 xp = *reinterpret_cast<const float2*>(src);
                    float x[3] = {xp.x, xp.y, 0.f}, dd[3];
                    if constexpr (NS) x[2] = src[64 - lane];
#pragma unroll
                    for (int v = 0; v < NV; ++v) dd[v] = fmaf(-a.tau32, r, fabsf(x[v]));
                    bool kp[3] = {dd[0] >= 0.f, dd[1] >= 0.f, NS && dd[2] >= 0.f};
                    const float db = delta * r;
                    float near_ = fminf(fabsf(dd[0]), fabsf(dd[1]));
                    if constexpr (NS) near_ = fminf(near_, fabsf(dd[2]));
                    if (__any_sync(FULL, near_ <= db)) {           // rare: recorded, and decided between the passes
                        BandRec& rc = rec[nrec++];
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            const bool in = fabsf(dd[v]) <= db;
                            const unsigned inb = __ballot_sync(FULL, in);
                            kp[v] = kp[v] && !in;
                            if (pass == 0) {
                                if (lane == 0) rc.lanes[v] = inb;
                                rc.d[v][lane] = dd[v];
                            } else {
                                kp[v] = kp[v] || ((rc.lanes[v] >> lane) & 1u) != 0u;
                            }
                        }
                        if (pass == 0 && lane == 0)
                            rc.head = (unsigned)(l == 0 || l == KB ? l : k0 + l) | ((unsigned)h0 << 8);
                    }
                    const int sl = l == 0 || l == KB ? l : k0 + l;          // in-place slot of the group
                    if (a.mask_out) {                               // words cleared before the launch
                        uint32_t* mo = a.mask_out + (size_t)grp * NBW + (sl == 0 ? 0 : (K >> e) + (sl >> e)) * (NF / 32);
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            const int f = C == 3 ? (h0 * 32 + lane) * 3 + v : v * 32 + lane;
                            if (kp[v]) atomicOr(&mo[f >> 5], 1u << (f & 31));
                        }
                    }
                    const float inv = __int_as_float((127 - e) << 23);      // 1 / support
                    if constexpr (ADJ) {                                    // r's coefficients take the place of x's
                        const float2 rp = *reinterpret_cast<const float2*>(src + ONE);
                        float rv[3] = {rp.x, rp.y, 0.f};
                        if constexpr (NS) rv[2] = src[ONE + 64 - lane];
#pragma unroll
                        for (int v = 0; v < NV; ++v) {
                            if (kp[v]) dot = fmaf(x[v] * inv, rv[v], dot);
                            x[v] = rv[v];
                        }
                    }
#pragma unroll
                    for (int hh = 0; hh < NH; ++hh) {
                        const bool mine = C == 3 ? (kp[0] || kp[1] || kp[2]) : kp[hh];
                        const unsigned bal = __ballot_sync(FULL, mine);    // (every lane has read its words)
                        if (bal == 0u) continue;
                        // basis rows of this half (8 lanes each) that keep a coefficient: bits 7, 15, 23, 31
                        const unsigned rb = (((bal & 0x7f7f7f7fu) + 0x7f7f7f7fu) | bal) & 0x80808080u;
                        const int rr = nrow + __popc(rb & below);
                        const float t0 = kp[hh] ? x[hh] * inv : 0.f;
                        float z0 = t0, zr = 0.f, zi = 0.f;
                        if constexpr (C == 3) {
                            const float t1 = kp[1] ? x[1] * inv : 0.f, t2 = kp[2] ? x[2] * inv : 0.f;
                            z0 = t0 + t1 + t2;
                            zr = t0 - 0.5f * (t1 + t2);
                            zi = G_S3H * (t2 - t1);
                            if (a.agg_mode) kept += (kp[0] ? 1 : 0) + (kp[1] ? 1 : 0) + (kp[2] ? 1 : 0);
                        } else {
                            if (a.agg_mode) kept += mine ? 1 : 0;
                        }
                        if (rb & rowbit) {
                            if (rr < cap) {
                                float* o = list + rr * G::RW + b;
                                o[0] = z0;
                                if constexpr (C == 3) {
                                    o[8] = zr;
                                    o[16] = zi;
                                }
                            } else {
                                float* o = spill + (rr - cap) * G::RW + b;
                                o[0] = z0;
                                if constexpr (C == 3) {
                                    o[8] = zr;
                                    o[16] = zi;
                                }
                            }
                        }
                        // row mask (bits 7, 15, 23, 31 -> 0 .. 3) and first row of the slot's half
                        const uint32_t info = ((rb * 0x00204081u) >> 28) | ((unsigned)nrow << 4);
                        if (lane == sl) slots |= info << (16 * (h0 + hh));
                        nrow += __popc(rb);
                    }
                }
                __syncwarp();
            }
        }
        dot_all = dot;
        if (left || pass == 1 || nrec == 0) break;
        __syncwarp();
        group_band<C, Tin>(a, rec, nrec, pnk, lin, lane);
        }
        if (left) break;
        if constexpr (ADJ) {
            dots += dot_all;
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) dots += __shfl_xor_sync(FULL, dots, off);
            if (lane == 0 && a.grad_w) a.grad_w[grp] = dots;
        }
        float wg = 1.f;
        if (a.w_in) wg = a.w_in[grp];
        else if (a.agg_mode == 1) wg = 1.f / (float)max(1, __reduce_add_sync(FULL, kept));
        if (lane == 0 && a.weights_out) a.weights_out[grp] = wg;
        __syncwarp();

        // the inverse; SP: part of the list is in the spill buffer
        auto inverse = [&](auto spilled) {
        constexpr bool SP = decltype(spilled)::value;
        // ---- stage D on the listed rows, in place: lane (p, b) of a step forms Z[row r0 + p][b]
        {
            float v0[PS], vr[PS], vi[PS];              // V_f[b][j], j = 0 .. 7
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float* vb = vt + b * PS + 4 * e;
                const float4 x = *reinterpret_cast<const float4*>(vb);
                v0[4 * e] = x.x; v0[4 * e + 1] = x.y; v0[4 * e + 2] = x.z; v0[4 * e + 3] = x.w;
                if constexpr (C == 3) {
                    const float4 y = *reinterpret_cast<const float4*>(vb + 64), z = *reinterpret_cast<const float4*>(vb + 128);
                    vr[4 * e] = y.x; vr[4 * e + 1] = y.y; vr[4 * e + 2] = y.z; vr[4 * e + 3] = y.w;
                    vi[4 * e] = z.x; vi[4 * e + 1] = z.y; vi[4 * e + 2] = z.z; vi[4 * e + 3] = z.w;
                }
            }
#pragma unroll 1
            for (int r0 = 0; r0 < nrow; r0 += 4) {
                const int r = r0 + (lane >> 3);
                const bool on = r < nrow;
                const int rc = on ? r : nrow - 1;
                float* row = list + rc * G::RW;
                if (SP && rc >= cap) row = spill + (rc - cap) * G::RW;
                float t[G::RW];
#pragma unroll
                for (int e = 0; e < G::RW / 4; ++e) {
                    const float4 x = reinterpret_cast<const float4*>(row)[e];
                    t[4 * e] = x.x; t[4 * e + 1] = x.y; t[4 * e + 2] = x.z; t[4 * e + 3] = x.w;
                }
                __syncwarp();
                float z0 = 0.f, zr = 0.f, zi = 0.f;
#pragma unroll
                for (int j = 0; j < PS; ++j) {
                    z0 = fmaf(t[j], v0[j], z0);
                    if constexpr (C == 3) {
                        zr = fmaf(t[8 + j], vr[j], fmaf(t[16 + j], vi[j], zr));
                        zi = fmaf(t[16 + j], vr[j], fmaf(-t[8 + j], vi[j], zi));
                    }
                }
                if (on) {
                    row[b] = z0;
                    if constexpr (C == 3) {
                        row[8 + b] = zr;
                        row[16 + b] = zi;
                    }
                }
            }
        }
        __syncwarp();
        if (q > 0)                                     // the accumulator of group q - 1 is final
            asm volatile("bar.sync %0, 64;" ::"r"(1 + (warp + GR_WARPS - 1) % GR_WARPS) : "memory");
        // ---- stage E, Haar synthesis and aggregation, depth first
        const Inverse<K, C, MF, SP> inv{slots, list + 2 * pb, spill + 2 * pb, cap, ut + pa * G::UF, acc + lane_off, aoff, wg,
                                            third, sq3, nsq3};
        inv.run();
        };
        if (!__any_sync(FULL, nrow > cap)) inverse(std::false_type());
        else inverse(std::true_type());
        if (q + 1 < ngr)                               // hand the accumulator to the warp of group q + 1
            asm volatile("bar.arrive %0, 64;" ::"r"(1 + warp) : "memory");
        grp = ahead;
    }
    __syncthreads();
    // the tile partial
    const int tile = ty * a.ntx + tx;
    if (2 * *probe > first) {
        if (tid == 0) A.counter[2 + atomicAdd(A.counter + 1, 1)] = tile;
        __syncthreads();
        return;
    }
    float* dst = a.partials + (size_t)tile * a.FHmax * a.FWmax * G::ACC;
    for (int r = warp; r < FH; r += GR_WARPS)
        for (int c = lane; c < FW; c += 32) {
            if constexpr (C == 3)
                reinterpret_cast<float4*>(dst)[r * a.FWmax + c] = reinterpret_cast<const float4*>(acc)[r * FWp + c];
            else
                reinterpret_cast<float2*>(dst)[r * a.FWmax + c] = reinterpret_cast<const float2*>(acc)[r * FWp + c];
        }
    __syncthreads();
}

// Persistent CTAs over the tiles of the band, in column stripes GR_STRIPE tiles wide: the planes'
// rows that the tiles in flight gather from then form a compact block that stays in L2.
constexpr int GR_STRIPE = 32;

template <int K, int C, typename Tin, bool MF, bool ADJ>
__global__ void __launch_bounds__(GR_THREADS, ADJ ? 4 : GR_CTAS) group_kernel(const __grid_constant__ GroupArgs A) {
    using G = GCfg<C>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ int item, probe;
    const FilterArgs& a = A.f;
    if (a.dense && *a.dense) return;
    float* ut = reinterpret_cast<float*>(smem);
    for (int t = threadIdx.x; t < PS2; t += GR_THREADS) {          // U table: [i][a], duplicated pairs
        const int i = t >> 3, r = t & 7;
        float* d = ut + t * G::UF;
        d[0] = d[1] = a.basis32[r * PS + i];
        if constexpr (C == 3) {
            const float ur = a.basis32[64 + r * PS + i], ui = a.basis32[128 + r * PS + i];
            d[2] = d[3] = ur;
            d[4] = d[5] = ui;
            d[6] = d[7] = -ui;
        }
    }
    float* vt = ut + PS2 * G::UF;                                   // V_0, V_1 (re, im): [b][j]
    for (int t = threadIdx.x; t < (C == 3 ? 3 : 1) * PS2; t += GR_THREADS) vt[t] = a.basis32[(C == 3 ? 192 : 64) + t];
    const int total = A.nty_band * a.ntx;
    float* spill = A.spill + (size_t)blockIdx.x * GR_WARPS * group_spill_warp(K, C);
    for (;;) {
        if (threadIdx.x == 0) item = atomicAdd(A.counter, 1);
        __syncthreads();
        const int w = __shfl_sync(0xffffffffu, item, 0);            // (uniform, as the warp index)
        __syncthreads();
        if (w >= total) break;
        const int per = GR_STRIPE * A.nty_band;
        const int st = w / per, r = w - st * per;
        const int sw = min(GR_STRIPE, a.ntx - st * GR_STRIPE);
        group_tile<K, C, Tin, MF, ADJ>(A, A.ty0 + r / sw, st * GR_STRIPE + r % sw, smem, spill, &probe);
    }
}

}  // namespace htsvd
