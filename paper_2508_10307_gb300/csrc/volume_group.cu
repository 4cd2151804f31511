// Volume filter on projection planes: Alg. 1 Steps 2(2)-(4) and 3 for the 4 x 4 x 4 cubes of a volume, after
// the image path's group filter (group_impl.cuh).
//
// * volume_plane_kernel: the projection of the cube at every position of a band of z planes, once (a position
//   belongs to four groups on average at K 32, stride 2). Warp = a row of positions; lane l = (basis row
//   i = l / 8, column j = l / 2 % 4, tube half l % 2) keeps a window of four Y_f columns in registers and
//   writes coefficients 2 l, 2 l + 1 of a position: 256 contiguous bytes.
// * volume_group_kernel: one warp per group. The pairs of all K cubes are gathered (coalesced), Haar analysed
//   in registers, thresholded slot by slot where one comparison cannot rule a slot out (FP64 inside the guard
//   band, decided between two passes), and the basis rows that kept a coefficient are listed in shared
//   memory after the tube DFT. Z_f = T_f V_f^H per listed row; then depth first over the Haar tree, U_f Z_f and the
//   inverse tube DFT per slot for the lane's two voxels, and each leaf is added to the CTA's footprint with
//   shared atomics. After the threshold a group keeps coefficients in a few of its 128 (slot, row) pairs, so
//   the inverse is a fraction of the dense one that volume_filter_kernel runs (5,900 warp instructions per
//   group).
//
// 176 x 208 x 176, stride 2, window 5, K 32 (780 K groups): 8.24 ms in volume_filter_kernel -> 0.48 (planes) + 4.21
// ms. The planes are bound by their stores (1.6 GB), the groups by instruction issue and shared memory latency at
// 16 warps per SM (128 registers; 8 warps share a footprint, since four footprints of 4-warp CTAs leave room for
// 12). volume_filter_kernel stays for small volumes and for windows whose footprint and row lists do not fit two
// CTAs per SM (window 6 at stride 3: 670 us either way on 32,768 references).
#include <algorithm>
#include <type_traits>

#include "f32x2.cuh"
#include "kernels.h"

namespace htsvd {

namespace {

constexpr int VE = 4;                   // cube edge
constexpr int VT = 4;                   // references per tile edge
constexpr int VG_WARPS = 8;
constexpr int VG_THREADS = VG_WARPS * 32;
constexpr int VG_RAW = 2;               // staged slots (64 floats) that fit behind a full row list
constexpr int VG_ROW = 16;              // floats per listed row: T_0, T_2, Re T_1, Im T_1 of four columns
constexpr unsigned ALL = 0xffffffffu;

__host__ __device__ inline int vpos(int i, int s, int n) {
    const int v = i * s, last = n - VE;
    return v < last ? v : last;
}

// ------------------------------------------------------------------------------ planes

__host__ __device__ constexpr int v_log2(int k) { return k <= 1 ? 0 : 1 + v_log2(k / 2); }
__host__ __device__ constexpr int v_ctz(int x) {
    return (x & 1) ? 0 : (x & 2) ? 1 : (x & 4) ? 2 : (x & 8) ? 3 : 4;
}
__host__ __device__ constexpr float v_root(int e) {
    return (e & 1) ? 1.41421356237309504880f * (float)(1 << (e >> 1)) : (float)(1 << (e >> 1));
}

// Rows of coefficients that VS_GROUPS groups spread over the volume keep, as sample_rows_kernel counts them for
// images: thread (cube k, basis row i) projects its row, 64 threads take the Haar transform of a coefficient each.
// The blocks of the first band's planes that come first do it, so that it costs no time of its own.
constexpr int VS_GROUPS = 128;

// Group b of the sample, by a block of 128 threads; sm: K * 64 floats, [k][i][j][tube].
template <int K>
__device__ __forceinline__ void volume_sample(const VolFilterArgs& A, int b, float* sm, unsigned* mask, int* st, int most) {
    const VolGeo& g = A.g;
    const int tid = threadIdx.x;
    const long long ng = (long long)g.nrz * g.nry * g.nrx;
    const long long grp = (2ll * b + 1) * ng / (2 * VS_GROUPS);
    if (tid < VE) mask[tid] = 0u;
    if (tid < K * VE) {
        const int k = tid >> 2, i = tid & 3;
        const uint8_t* cube = A.vol + A.idx[grp * K + k];
        const size_t plane = (size_t)g.H * g.W;
        const double *U = A.basis64, *V = A.basis64 + 4 * 16 * 2;      // [slice][a * 4 + i][re, im]
        float y0[VE] = {}, y2[VE] = {}, yr[VE] = {}, yi[VE] = {};
#pragma unroll
        for (int a = 0; a < VE; ++a) {
            const float u0 = (float)U[(a * 4 + i) * 2], u2 = (float)U[(32 + a * 4 + i) * 2];
            const float ur = (float)U[(16 + a * 4 + i) * 2], ui = (float)U[(16 + a * 4 + i) * 2 + 1];
#pragma unroll
            for (int b = 0; b < VE; ++b) {
                const uint8_t* p = cube + (size_t)a * g.W + b;
                const float p0 = p[0], p1 = p[plane], p2 = p[2 * plane], p3 = p[3 * plane];
                const float Xr = p0 - p2, Xi = p3 - p1;
                y0[b] = fmaf(u0, (p0 + p1) + (p2 + p3), y0[b]);
                y2[b] = fmaf(u2, (p0 - p1) + (p2 - p3), y2[b]);
                yr[b] = fmaf(ur, Xr, fmaf(ui, Xi, yr[b]));
                yi[b] = fmaf(ur, Xi, fmaf(-ui, Xr, yi[b]));
            }
        }
        float* d = sm + tid * 16;
#pragma unroll
        for (int j = 0; j < VE; ++j) {
            float z0 = 0.f, z2 = 0.f, zr = 0.f, zi = 0.f;
#pragma unroll
            for (int b = 0; b < VE; ++b) {
                const float vr = (float)V[(16 + b * 4 + j) * 2], vi = (float)V[(16 + b * 4 + j) * 2 + 1];
                z0 = fmaf(y0[b], (float)V[(b * 4 + j) * 2], z0);
                z2 = fmaf(y2[b], (float)V[(32 + b * 4 + j) * 2], z2);
                zr = fmaf(yr[b], vr, fmaf(-yi[b], vi, zr));
                zi = fmaf(yr[b], vi, fmaf(yi[b], vr, zi));
            }
            d[j * 4] = 0.25f * fmaf(2.f, zr, z0 + z2);
            d[j * 4 + 1] = 0.25f * fmaf(-2.f, zi, z0 - z2);
            d[j * 4 + 2] = 0.25f * fmaf(-2.f, zr, z0 + z2);
            d[j * 4 + 3] = 0.25f * fmaf(2.f, zi, z0 - z2);
        }
    }
    __syncthreads();
    if (tid < 64) {
        float p[K];
#pragma unroll
        for (int k = 0; k < K; ++k) p[k] = sm[k * 64 + tid];
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
            if (fabsf(p[l]) >= A.tau32 * v_root(l == 0 ? v_log2(K) : v_ctz(l) + 1)) keep |= 1u << l;
        atomicOr(&mask[tid >> 4], keep);
    }
    __syncthreads();
    if (tid == 0) {
        int rows = 0;
        for (int i = 0; i < VE; ++i) rows += __popc(mask[i]);
        atomicAdd(st, rows);
        __threadfence();
        if (atomicAdd(st + 1, 1) == VS_GROUPS - 1) st[2] = atomicAdd(st, 0) > most * VS_GROUPS;
    }
}

constexpr int VP_NX = 61;               // positions per CTA row (64 columns)
constexpr int VP_NY = 4;

// SK: slots of the groups that the first zs slices of blocks sample (0: no such slices).
template <int SK>
__global__ void __launch_bounds__(128, 4) volume_plane_kernel(const __grid_constant__ VolPlaneArgs a,
                                                           const __grid_constant__ VolFilterArgs f, int zs, int most) {
    __shared__ __align__(16) float ub[3][2][16];                      // [slice][re, im][a * 4 + i]
    __shared__ __align__(16) float yb[VP_NY][64][4][4];               // [y][x][i][Y_0, Y_2, Re Y_1, Im Y_1]
    __shared__ float qs[VP_NY][64];
    __shared__ uint8_t px[VE][VP_NY + VE - 1][64];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int npx = a.W - VE + 1, npy = a.H - VE + 1;
    if constexpr (SK > 0) {
        if ((int)blockIdx.z < zs) {
            const int b = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
            if (b < VS_GROUPS) volume_sample<SK>(f, b, &yb[0][0][0][0], reinterpret_cast<unsigned*>(qs), a.sample, most);
            return;
        }
    }
    // (by now known to be dense: nobody reads the planes)
    if (a.sample && __syncthreads_or(threadIdx.x == 0 && *(volatile int*)(a.sample + 2))) return;
    const int zb = blockIdx.z - zs;
    const int x0 = blockIdx.x * VP_NX, y0 = blockIdx.y * VP_NY, z = a.pz0 + zb;
    if (tid < 96) {
        const int f = tid / 32, ri = (tid >> 4) & 1, ai = tid & 15;
        ub[f][ri][ai] = (float)a.basis64[((size_t)f * 16 + ai) * 2 + ri];
    }
    for (int t = tid; t < VE * (VP_NY + VE - 1) * 64; t += 128) {
        const int c = t / ((VP_NY + VE - 1) * 64), r = t / 64 % (VP_NY + VE - 1), x = t & 63;
        px[c][r][x] = (y0 + r < a.H && x0 + x < a.W)
                          ? a.vol[((size_t)(z + c) * a.H + y0 + r) * a.W + x0 + x] : (uint8_t)0;
    }
    __syncthreads();
#pragma unroll 1
    for (int t = tid; t < VP_NY * 64; t += 128) {
        const int y = t >> 6, x = t & 63;
        float s0[4] = {}, s2[4] = {}, sr[4] = {}, si[4] = {}, q = 0.f;
#pragma unroll
        for (int r = 0; r < VE; ++r) {
            const float p0 = px[0][y + r][x], p1 = px[1][y + r][x], p2 = px[2][y + r][x], p3 = px[3][y + r][x];
            q = fmaf(p0, p0, fmaf(p1, p1, fmaf(p2, p2, fmaf(p3, p3, q))));
            const float X0 = (p0 + p1) + (p2 + p3), X2 = (p0 - p1) + (p2 - p3), Xr = p0 - p2, Xi = p3 - p1;
            const float4 u0 = *reinterpret_cast<const float4*>(&ub[0][0][r * 4]), u2 = *reinterpret_cast<const float4*>(&ub[2][0][r * 4]);
            const float4 ur = *reinterpret_cast<const float4*>(&ub[1][0][r * 4]), ui = *reinterpret_cast<const float4*>(&ub[1][1][r * 4]);
            const float U0[4] = {u0.x, u0.y, u0.z, u0.w}, U2[4] = {u2.x, u2.y, u2.z, u2.w};
            const float UR[4] = {ur.x, ur.y, ur.z, ur.w}, UI[4] = {ui.x, ui.y, ui.z, ui.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                s0[i] = fmaf(U0[i], X0, s0[i]);
                s2[i] = fmaf(U2[i], X2, s2[i]);
                sr[i] = fmaf(UR[i], Xr, fmaf(UI[i], Xi, sr[i]));
                si[i] = fmaf(UR[i], Xi, fmaf(-UI[i], Xr, si[i]));
            }
        }
        qs[y][x] = q;
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(yb[y][x][i]) = make_float4(s0[i], s2[i], sr[i], si[i]);
    }
    __syncthreads();
    const int nx = min(VP_NX, npx - x0), ny = min(VP_NY, npy - y0);
    const size_t row0 = ((size_t)zb * npy + y0) * npx + x0;
    for (int t = tid; t < ny * VP_NX; t += 128) {
        const int y = t / VP_NX, x = t - y * VP_NX;
        if (x < nx) a.pn[row0 + (size_t)y * npx + x] = (qs[y][x] + qs[y][x + 1]) + (qs[y][x + 2] + qs[y][x + 3]);
    }
    if (warp >= ny) return;
    const int i = lane >> 3, j = (lane >> 1) & 3, kp = lane & 1;
    float v0[4], v2[4], vr[4], vi[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const double* V = a.basis64 + ((size_t)4 * 16 + b * 4 + j) * 2;
        v0[b] = (float)V[0];
        vr[b] = (float)V[32];
        vi[b] = (float)V[33];
        v2[b] = (float)V[64];
    }
    float4 w[4];
    float* dst = a.coef + (row0 + (size_t)warp * npx) * 64 + lane * 2;
#pragma unroll
    for (int b = 0; b < 3; ++b) w[b] = *reinterpret_cast<const float4*>(yb[warp][b][i]);
#pragma unroll 1
    for (int xb = 0; xb < nx; xb += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int x = xb + u;
            if (x < nx) {                              // warp-uniform
                w[(u + 3) & 3] = *reinterpret_cast<const float4*>(yb[warp][x + 3][i]);
                float z0 = 0.f, z2 = 0.f, zr = 0.f, zi = 0.f;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const float4 y = w[(u + b) & 3];
                    z0 = fmaf(y.x, v0[b], z0);
                    z2 = fmaf(y.y, v2[b], z2);
                    zr = fmaf(y.z, vr[b], fmaf(-y.w, vi[b], zr));
                    zi = fmaf(y.z, vi[b], fmaf(y.w, vr[b], zi));
                }
                // tube 0, 1 (kp = 0) or 2, 3: (z0 + z2 +- 2 zr) / 4, (z0 - z2 -+ 2 zi) / 4
                const float s = kp ? -2.f : 2.f;
                *reinterpret_cast<float2*>(dst + (size_t)x * 64) =
                    make_float2(0.25f * fmaf(s, zr, z0 + z2), 0.25f * fmaf(-s, zi, z0 - z2));
            }
        }
}

// ------------------------------------------------------------------------------ group filter

struct VolSm {
    __align__(16) float u[4][2][4][4];  // [i][tube half][a][U_0, U_2, +- U_1r, -U_1i]
    __align__(16) float v[4][4][4];     // [b][V_0, V_2, V_1r, V_1i][j]
    double ud[2][3][2][16];             // [U, V][slice][re, im][a * 4 + i]
};

// Guard-band record of a Haar slot (global scratch).
struct VolRec {
    uint32_t slot, lanes[2];
};

// FP64 coefficient e = (i * 4 + j) * 4 + k of the cube at position lin.
__device__ __noinline__ double vol_coef64(const VolFilterArgs& A, const VolSm& sm, int lin, int e) {
    const int i = e >> 4, j = (e >> 2) & 3, k = e & 3;
    const size_t plane = (size_t)A.g.H * A.g.W;
    double t0 = 0, t2 = 0, t1r = 0, t1i = 0;
    for (int a = 0; a < 4; ++a)
        for (int b = 0; b < 4; ++b) {
            const uint8_t* p = A.vol + lin + (size_t)a * A.g.W + b;
            const double p0 = p[0], p1 = p[plane], p2 = p[2 * plane], p3 = p[3 * plane];
            const double x0 = p0 + p1 + p2 + p3, x2 = p0 - p1 + p2 - p3, xr = p0 - p2, xi = p3 - p1;
            const double u0 = sm.ud[0][0][0][a * 4 + i], v0 = sm.ud[1][0][0][b * 4 + j];
            const double u2 = sm.ud[0][2][0][a * 4 + i], v2 = sm.ud[1][2][0][b * 4 + j];
            t0 += u0 * x0 * v0;
            t2 += u2 * x2 * v2;
            const double ur = sm.ud[0][1][0][a * 4 + i], ui = sm.ud[0][1][1][a * 4 + i];
            const double vr = sm.ud[1][1][0][b * 4 + j], vi = sm.ud[1][1][1][b * 4 + j];
            const double yr = ur * xr + ui * xi, yi = ur * xi - ui * xr;          // conj(u) x
            t1r += yr * vr - yi * vi;
            t1i += yr * vi + yi * vr;
        }
    const double sg = (k & 1) ? -1.0 : 1.0;
    const double c1 = k == 0 ? 2 * t1r : k == 1 ? -2 * t1i : k == 2 ? -2 * t1r : 2 * t1i;
    return 0.25 * (t0 + sg * t2 + c1);
}

// Replaces the lanes of each record by those that keep their coefficient (lane k forms cube k's coefficient,
// the Haar row weighs the cubes).
__device__ __noinline__ void vol_band(const VolFilterArgs& A, const VolSm& sm, VolRec* rec, int n, int lin, int lane) {
    const int K = A.g.K;
    for (int r = 0; r < n; ++r) {
        const int sl = (int)rec[r].slot, st = sl == 0 ? K : 1 << (__ffs(sl) - 1);   // half support
        const double mag = 1.0 / sqrt((double)(sl == 0 ? K : 2 * st));
        double h = 0.0;
        if (lane < K) {
            if (sl == 0) h = mag;
            else if (lane >= sl - st && lane < sl) h = mag;
            else if (lane >= sl && lane < sl + st) h = -mag;
        }
        for (int v = 0; v < 2; ++v) {
            uint32_t open = rec[r].lanes[v], keep = 0;
            while (open) {
                const int l = __ffs(open) - 1;
                open &= open - 1;
                double t = h != 0.0 ? h * vol_coef64(A, sm, lin, 2 * l + v) : 0.0;
                for (int o = 16; o >= 1; o >>= 1) t += __shfl_xor_sync(ALL, t, o);
                if (fabs(t) >= A.tau64) keep |= 1u << l;
            }
            if (lane == 0) rec[r].lanes[v] = keep;
        }
    }
    __syncwarp();
}

// The inverse of one group from its row list (rows already through V^H).
template <int K>
struct VolInverse {
    static constexpr int LV = v_log2(K);
    uint32_t slots;          // lane sl: row mask | first row << 4
    const float* z;          // row list + the lane's column (b)
    int hoff, goff;          // offsets of the two rows of Z_1 in the lane's order
    const float* u;          // U table of the lane's voxels
    float sg2;               // +1, -1: g0 +- g2
    float* num;              // footprint + the lane's first voxel
    int dk;                  // distance of its second voxel
    int voff;                // lane k: footprint offset of cube k
    float wgt;

    __device__ __forceinline__ f2 value(int sl) const {
        const uint32_t word = __shfl_sync(ALL, slots, sl);
        if (word == 0u) return 0;                      // warp-uniform
        float s = 0.f, g2 = 0.f, g = 0.f;
        const float* row = z + (word >> 4) * VG_ROW;
#pragma unroll 1
        for (uint32_t m = word & 15u; m; m &= m - 1, row += VG_ROW) {
            const float4 q = *reinterpret_cast<const float4*>(u + (__ffs(m) - 1) * 32);
            s = fmaf(q.x, row[0], s);
            g2 = fmaf(q.y, row[4], g2);
            g = fmaf(q.z, row[hoff], fmaf(q.w, row[goff], g));
        }
        s = fmaf(sg2, g2, s);
        return f2_mul(f2_pack(fmaf(2.f, g, s), fmaf(-2.f, g, s)), f2_dup(0.25f));
    }
    __device__ __forceinline__ void leaf(int k, f2 v) const {
        const int off = __shfl_sync(ALL, voff, k);
        float a, b;
        f2_unpack(v, a, b);
        atomicAdd(num + off, wgt * a);
        atomicAdd(num + off + dk, wgt * b);
    }
    template <int l>
    __device__ __forceinline__ void node(int idx, f2 v) const {
        if constexpr (l == LV) {
            leaf(idx, v);
        } else {
            const f2 d = value((2 * idx + 1) * (K >> (l + 1)));
            node<l + 1>(2 * idx, f2_add(v, d));
            node<l + 1>(2 * idx + 1, f2_sub(v, d));
        }
    }
    __device__ __forceinline__ void run() const {
        constexpr int TL = LV > 2 ? LV - 2 : 0;
        const f2 root = value(0);
        f2 d[TL > 0 ? TL : 1];
#pragma unroll 1
        for (int t = 0; t < (1 << TL); ++t) {
            f2 v = root;
#pragma unroll
            for (int i = 0; i < TL; ++i) {
                if ((t & ((1 << (TL - i)) - 1)) == 0) d[i] = value((2 * (t >> (TL - i)) + 1) * (K >> (i + 1)));
                v = f2_fma(f2_dup(((t >> (TL - 1 - i)) & 1) ? -1.f : 1.f), d[i], v);
            }
            node<TL>(t, v);
        }
    }
};

__device__ __forceinline__ f2 vol_ldg(const float* p) {
    f2 v;
    asm volatile("ld.global.nc.b64 %0, [%1];" : "=l"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ void vol_stage(uint32_t mask, uint32_t bit, uint32_t& d, f2 pair) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b32 t;\n\tand.b32 t, %1, %2;\n\tsetp.ne.b32 p, t, 0;\n\t"
        "@p st.shared.b64 [%0], %3;\n\t@p add.u32 %0, %0, 256;\n\t}"
        : "+r"(d)
        : "r"(mask), "r"(bit), "l"(pair)
        : "memory");
}

struct VolLayout {
    int pos, list, num, total;
};
__host__ __device__ inline VolLayout vol_layout(int nvox, int cap) {
    VolLayout L;
    int o = 0;
    L.pos = o; o += VG_WARPS * 32 * 4;
    const int rows = VG_WARPS * (cap * VG_ROW + VG_RAW * 64);      // reused by the box sum after the last group
    L.list = o; o += (rows > nvox ? rows : nvox) * 4;
    L.num = o; o += 2 * nvox * 4;                      // numerator, origin weights
    L.total = o;
    return L;
}

template <int K>
__global__ void __launch_bounds__(VG_THREADS, 2) volume_group_kernel(const __grid_constant__ VolGroupArgs G) {
    constexpr int LV = v_log2(K), CAP = K * 4;         // every row of every slot fits
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ VolSm sm;
    const VolFilterArgs& A = G.f;
    if (A.dense && *A.dense) return;
    const VolGeo& g = A.g;
    const int tid = threadIdx.x, warp = __shfl_sync(ALL, tid >> 5, 0), lane = tid & 31;
    // tile of references and its footprint
    const int nty = (g.nry + VT - 1) / VT, ntx = (g.nrx + VT - 1) / VT;
    const int tz = G.tz0 + blockIdx.x / (nty * ntx), trem = blockIdx.x % (nty * ntx);
    const int ty = trem / ntx, tx = trem - ty * ntx;
    int f0[3], fn[3];
    {
        const int t3[3] = {tz, ty, tx}, nr[3] = {g.nrz, g.nry, g.nrx}, nn[3] = {g.D, g.H, g.W};
        const int np[3] = {g.npz, g.npy, g.npx}, wl[3] = {g.wnz, g.wny, g.wnx};
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const int r0 = t3[d] * VT, r1 = min(r0 + VT, nr[d]) - 1;
            f0[d] = win_start(vpos(r0, g.s, nn[d]), np[d], g.win);
            fn[d] = win_start(vpos(r1, g.s, nn[d]), np[d], g.win) + wl[d] + VE - 1 - f0[d];
        }
    }
    const int nvox = fn[0] * fn[1] * fn[2];
    const VolLayout L = vol_layout(nvox, CAP);
    uint32_t* posw = reinterpret_cast<uint32_t*>(dyn + L.pos) + warp * 32;
    float* list = reinterpret_cast<float*>(dyn + L.list) + warp * (CAP * VG_ROW + VG_RAW * 64);
    float* num = reinterpret_cast<float*>(dyn + L.num);
    float* org = num + nvox;
    float* tmp = reinterpret_cast<float*>(dyn + L.list);
    for (int e = tid; e < 2 * 3 * 2 * 16; e += VG_THREADS) {
        const int w = e / 96, f = (e / 32) % 3, ri = (e / 16) & 1, ai = e & 15;
        const double v = A.basis64[((w * 4 + f) * 16 + ai) * 2 + ri];
        sm.ud[w][f][ri][ai] = v;
        const int a = ai >> 2, i = ai & 3;
        if (w == 0) {                                  // tube half 0 takes Re (u z), half 1 -Im (u z)
            if (f == 0) sm.u[i][0][a][0] = sm.u[i][1][a][0] = (float)v;
            if (f == 2) sm.u[i][0][a][1] = sm.u[i][1][a][1] = (float)v;
            if (f == 1 && ri == 0) {
                sm.u[i][0][a][2] = (float)v;
                sm.u[i][1][a][2] = -(float)v;
            }
            if (f == 1 && ri == 1) sm.u[i][0][a][3] = sm.u[i][1][a][3] = -(float)v;
        } else {
            if (f == 0 && ri == 0) sm.v[a][0][i] = (float)v;
            if (f == 2 && ri == 0) sm.v[a][1][i] = (float)v;
            if (f == 1) sm.v[a][2 + ri][i] = (float)v;
        }
    }
    for (int q = tid; q < 2 * nvox; q += VG_THREADS) num[q] = 0.f;
    __syncthreads();

    const int plane = g.H * g.W;
    const int r0z = tz * VT, r0y = ty * VT, r0x = tx * VT;
    const int nz = min(VT, g.nrz - r0z), ny = min(VT, g.nry - r0y), nx = min(VT, g.nrx - r0x);
    const int ngr = nz * ny * nx;
    // stage D: lane = (row of eight, column b); inverse: lane = (row a, column b, tube half)
    const int db = lane & 3;
    const int ea = lane >> 3, eb = (lane >> 1) & 3, eh = lane & 1;
    const int lane_vox = (eh * fn[1] + ea) * fn[2] + eb;       // voxel k = eh, second one two slices on
    const unsigned rowbit = 0x80u << (lane & 24), below = (1u << (lane & 24)) - 1u;
    const int kp = lane & 1, jj = (lane >> 1) & 3;
    float rtab = 1.f;
#pragma unroll
    for (int e = 1; e < 6; ++e) rtab = lane == e ? v_root(e) : rtab;
    VolRec* rec = reinterpret_cast<VolRec*>(G.rec) + ((size_t)blockIdx.x * VG_WARPS + warp) * 32;

#pragma unroll 1
    for (int q = warp; q < ngr; q += VG_WARPS) {
        const int qz = q / (ny * nx), qr = q - qz * (ny * nx), qy = qr / nx, qx = qr - qy * nx;
        const size_t gi = ((size_t)(r0z + qz) * g.nry + (r0y + qy)) * g.nrx + (r0x + qx);
        int lin = 0, voff = 0;
        float pnk = 0.f;
        uint32_t ppos = 0;
        if (lane < K) {
            lin = A.idx[gi * K + lane];
            const int cz = lin / plane, crem = lin - cz * plane;
            const int cy = crem / g.W, cx = crem - cy * g.W;
            voff = ((cz - f0[0]) * fn[1] + cy - f0[1]) * fn[2] + cx - f0[2];
            ppos = (uint32_t)(((cz - G.pz0) * g.npy + cy) * g.npx + cx);
            pnk = G.pn[ppos];
        }
        posw[lane] = ppos;
        __syncwarp();
        float nrm2 = pnk;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) nrm2 += __shfl_xor_sync(ALL, nrm2, o);
        const float delta = A.band_rel * sqrtf(nrm2) + A.band_abs;
        const float lo1 = (A.tau32 - delta) * (1.f - 1e-6f) - 1e-30f;
        int nrow = 0, kept = 0;
        uint32_t slots = 0;
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            int nrec = 0;
            nrow = kept = 0;
            slots = 0;
            // ---- gather and Haar analysis (unnormalised, in place)
            f2 p[K];
            {
                const float* src = G.coef + lane * 2;
                if constexpr (K >= 4) {
#pragma unroll
                    for (int k = 0; k < K; k += 4) {
                        const uint4 o = *reinterpret_cast<const uint4*>(posw + k);
                        p[k] = vol_ldg(src + (size_t)o.x * 64);
                        p[k + 1] = vol_ldg(src + (size_t)o.y * 64);
                        p[k + 2] = vol_ldg(src + (size_t)o.z * 64);
                        p[k + 3] = vol_ldg(src + (size_t)o.w * 64);
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < K; ++k) p[k] = vol_ldg(src + (size_t)posw[k] * 64);
                }
            }
#pragma unroll
            for (int d = 1; d < K; d <<= 1)
#pragma unroll
                for (int m = 0; m < K; m += 2 * d) {
                    const f2 x = p[m], y = p[m + d];
                    p[m + d] = f2_sub(x, y);
                    p[m] = f2_add(x, y);
                }
            // ---- slots where some lane may keep a coefficient
            uint32_t act = 0;
            float lo[LV + 1];
#pragma unroll
            for (int e = 1; e <= LV; ++e) lo[e] = lo1 * v_root(e);
#pragma unroll
            for (int l = 0; l < K; ++l) {
                const float mx = fmaxf(fabsf(f2_lo(p[l])), fabsf(f2_hi(p[l])));
                if (!(mx < lo[l == 0 ? LV : v_ctz(l) + 1])) act |= 1u << l;
            }
            act = __reduce_or_sync(ALL, act);
            // ---- threshold, a batch of slots at a time (staged behind the list, as in group_impl.cuh)
#pragma unroll 1
            while (act) {
                float* raw = list + nrow * VG_ROW;
                const int room = (CAP - nrow) * VG_ROW / 64 + VG_RAW;
                uint32_t sub = act;
                if (__popc(act) > room) sub = act & ((2u << __fns(act, 0, room)) - 1u);
                act &= ~sub;
                uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(raw + lane * 2));
#pragma unroll
                for (int l = 0; l < K; ++l) vol_stage(sub, 1u << l, d, p[l]);
                __syncwarp();
                const float* src = raw + lane * 2;
#pragma unroll 1
                for (; sub; sub &= sub - 1, src += 64) {
                    const int sl = __ffs(sub) - 1;
                    const int e = sl == 0 ? LV : __ffs(sl);                 // support 2^e
                    const float r = __shfl_sync(ALL, rtab, e);
                    const float2 x = *reinterpret_cast<const float2*>(src);
                    const float da = fmaf(-A.tau32, r, fabsf(x.x)), dc = fmaf(-A.tau32, r, fabsf(x.y));
                    bool ka = da >= 0.f, kc = dc >= 0.f;
                    const float db_ = delta * r;
                    if (__any_sync(ALL, fminf(fabsf(da), fabsf(dc)) <= db_)) {   // rare
                        VolRec& rc = rec[nrec++];
                        const bool ia = fabsf(da) <= db_, ic = fabsf(dc) <= db_;
                        const unsigned ma = __ballot_sync(ALL, ia), mc = __ballot_sync(ALL, ic);
                        ka = ka && !ia;
                        kc = kc && !ic;
                        if (pass == 0) {
                            if (lane == 0) {
                                rc.slot = (uint32_t)sl;
                                rc.lanes[0] = ma;
                                rc.lanes[1] = mc;
                            }
                        } else {
                            ka = ka || ((rc.lanes[0] >> lane) & 1u) != 0u;
                            kc = kc || ((rc.lanes[1] >> lane) & 1u) != 0u;
                        }
                    }
                    if (A.mask_out) {                               // words cleared before the launch
                        uint32_t* mo = A.mask_out + gi * 2 * K + 2 * (sl == 0 ? 0 : (K >> e) + (sl >> e)) + (lane >> 4);
                        const unsigned bits = (ka ? 1u : 0u) | (kc ? 2u : 0u);
                        if (bits) atomicOr(mo, bits << ((2 * lane) & 31));
                    }
                    const unsigned bal = __ballot_sync(ALL, ka || kc);     // (every lane has read its words)
                    if (bal == 0u) continue;
                    if (A.agg_mode) kept += (ka ? 1 : 0) + (kc ? 1 : 0);
                    // basis rows (8 lanes each) that keep a coefficient: bits 7, 15, 23, 31
                    const unsigned rb = (((bal & 0x7f7f7f7fu) + 0x7f7f7f7fu) | bal) & 0x80808080u;
                    // tube DFT of (s0, s1 | s2, s3), held by neighbouring lanes
                    const float inv = __int_as_float((127 - e) << 23);
                    const float a = ka ? x.x * inv : 0.f, b = kc ? x.y * inv : 0.f;
                    const float t1 = kp ? a + b : a - b, t2 = kp ? a : b;
                    const float o1 = __shfl_xor_sync(ALL, t1, 1), o2 = __shfl_xor_sync(ALL, t2, 1);
                    if (rb & rowbit) {
                        float* o = list + (nrow + __popc(rb & below)) * VG_ROW + kp * 4 + jj;
                        o[0] = (kp ? a - b : a + b) + o1;                    // T_0 | T_2
                        o[8] = kp ? b - o2 : a - o2;                         // Re T_1 | Im T_1
                    }
                    if (lane == sl) slots = ((rb * 0x00204081u) >> 28) | ((unsigned)nrow << 4);
                    nrow += __popc(rb);
                }
                __syncwarp();
            }
            if (pass == 1 || nrec == 0) break;
            __syncwarp();
            vol_band(A, sm, rec, nrec, lin, lane);
        }
        float wgt = 1.f;
        if (A.w_in) wgt = A.w_in[gi];
        else if (A.agg_mode == 1) wgt = 1.f / (float)max(1, __reduce_add_sync(ALL, kept));
        if (lane == 0 && A.weights_out) A.weights_out[gi] = wgt;
        // ---- Z_f[i, :] = T_f[i, :] V_f^H on the listed rows, eight at a time, in place
        {
            const float4 v0 = *reinterpret_cast<const float4*>(sm.v[db][0]), v2 = *reinterpret_cast<const float4*>(sm.v[db][1]);
            const float4 vr = *reinterpret_cast<const float4*>(sm.v[db][2]), vi = *reinterpret_cast<const float4*>(sm.v[db][3]);
#pragma unroll 1
            for (int r8 = 0; r8 < nrow; r8 += 8) {
                const int r = r8 + (lane >> 2);
                float* row = list + min(r, nrow - 1) * VG_ROW;
                const float4 t0 = reinterpret_cast<const float4*>(row)[0], t2 = reinterpret_cast<const float4*>(row)[1];
                const float4 tr = reinterpret_cast<const float4*>(row)[2], ti = reinterpret_cast<const float4*>(row)[3];
                __syncwarp();
                const float z0 = fmaf(t0.w, v0.w, fmaf(t0.z, v0.z, fmaf(t0.y, v0.y, t0.x * v0.x)));
                const float z2 = fmaf(t2.w, v2.w, fmaf(t2.z, v2.z, fmaf(t2.y, v2.y, t2.x * v2.x)));
                float zr = tr.x * vr.x, zi = ti.x * vr.x;              // t conj(v)
                zr = fmaf(ti.x, vi.x, zr); zi = fmaf(-tr.x, vi.x, zi);
                zr = fmaf(tr.y, vr.y, fmaf(ti.y, vi.y, zr)); zi = fmaf(ti.y, vr.y, fmaf(-tr.y, vi.y, zi));
                zr = fmaf(tr.z, vr.z, fmaf(ti.z, vi.z, zr)); zi = fmaf(ti.z, vr.z, fmaf(-tr.z, vi.z, zi));
                zr = fmaf(tr.w, vr.w, fmaf(ti.w, vi.w, zr)); zi = fmaf(ti.w, vr.w, fmaf(-tr.w, vi.w, zi));
                if (r < nrow) {
                    row[db] = z0;
                    row[4 + db] = z2;
                    row[8 + db] = zr;
                    row[12 + db] = zi;
                }
            }
        }
        __syncwarp();
        // ---- slot values, Haar synthesis, aggregation. Half 0: Re(u z) = ur zr - ui zi; half 1:
        //      -Im(u z) = -ur zi - ui zr
        const VolInverse<K> in{slots, list + eb, eh ? 12 : 8, eh ? 8 : 12, &sm.u[0][eh][ea][0], eh ? -1.f : 1.f,
                               num + lane_vox, 2 * fn[1] * fn[2], voff, wgt};
        in.run();
        if (lane < K) atomicAdd(org + voff, wgt);
        __syncwarp();
    }
    __syncthreads();
    // denominator: the weights of every cube covering a voxel = a 4 x 4 x 4 box sum of the origin weights
    for (int q = tid; q < nvox; q += VG_THREADS) {                 // along x
        const int xx = q % fn[2];
        float s = 0.f;
        for (int d = 0; d < 4 && d <= xx; ++d) s += org[q - d];
        tmp[q] = s;
    }
    __syncthreads();
    for (int q = tid; q < nvox; q += VG_THREADS) {                 // along y
        const int yy = (q / fn[2]) % fn[1];
        float s = 0.f;
        for (int d = 0; d < 4 && d <= yy; ++d) s += tmp[q - d * fn[2]];
        org[q] = s;
    }
    __syncthreads();
    for (int q = tid; q < nvox; q += VG_THREADS) {                 // along z, then into the volume
        const int zz = q / (fn[1] * fn[2]);
        float d = 0.f;
        for (int k = 0; k < 4 && k <= zz; ++k) d += org[q - k * fn[1] * fn[2]];
        if (d == 0.f) continue;
        const int rem = q - zz * (fn[1] * fn[2]);
        const int yy = rem / fn[2], xx = rem - yy * fn[2];
        const long long o = (long long)(f0[0] + zz) * plane + (long long)(f0[1] + yy) * g.W + f0[2] + xx;
        atomicAdd(A.num + o, num[q]);
        atomicAdd(A.den + o, d);
    }
}

// Voxels of a tile's footprint, at most a million (in 64 bits: strides of a few hundred pass 2^31).
int vol_nvox(const VolGeo& g) {
    const int ext[3] = {g.wnz, g.wny, g.wnx};
    int64_t n = 1;
    for (int d = 0; d < 3; ++d) n = std::min<int64_t>(n * ((int64_t)(VT - 1) * g.s + ext[d] + VE - 1), 1 << 20);
    return (int)n;
}

template <int K>
cudaError_t launch_vg(const VolGroupArgs& a, int tiles, cudaStream_t s) {
    const int smem = vol_layout(vol_nvox(a.f.g), K * 4).total;
    auto fn = volume_group_kernel<K>;
    cudaError_t e = allow_smem(fn, 3072);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    fn<<<tiles, VG_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

bool volume_group_fits(const VolGeo& g) {
    return vol_layout(vol_nvox(g), g.K * 4).total <= 110 * 1024 && g.H / VP_NY <= 65535;
}

// us of the filter with its planes against volume_filter_kernel, window 5, K 32, by the rows kept per group: 7,600
// references 178 / 198 at 10, 215 / 205 at 17, 408 / 333 at 64; 31,744: 484 / 540 at 26, 581 / 583 at 38, 1,386 / 1,068
// at 112; 120,050: 1,782 / 1,978 at 38, 2,363 / 2,314 at 64, 7,124 / 5,253 at 127. K 16: 165 / 166 at 18, 393 / 412 at
// 30, 604 / 540 at 55; 1,214 / 1,380 at 30, 1,801 / 1,732 at 54. (Leaving single tiles to the other kernel, as images
// do, took 447 us at 7,600 references and 26 rows, since each kernel waits for its last tiles, and the registers it
// needed cost 7 % everywhere.) With 8 slots or fewer: at any.
int volume_rows_limit(const VolGeo& g) {
    const int64_t ng = (int64_t)g.nrz * g.nry * g.nrx;
    if (g.K <= 8 || !volume_filter_fits(g)) return kEveryRow;
    if (g.K == 32) return ng < 15000 ? 14 : ng < 60000 ? 38 : 62;
    return ng < 15000 ? 18 : ng < 60000 ? 36 : 47;
}

int volume_tiles_z(const VolGeo& g) { return (g.nrz + VT - 1) / VT; }

int volume_tiles_plane(const VolGeo& g) { return ((g.nry + VT - 1) / VT) * ((g.nrx + VT - 1) / VT); }

void volume_band(const VolGeo& g, int t0, int t1, int& z0, int& z1) {
    z0 = win_start(vpos(t0 * VT, g.s, g.D), g.npz, g.win);
    z1 = win_start(vpos(std::min(t1 * VT, g.nrz) - 1, g.s, g.D), g.npz, g.win) + g.wnz;
}

size_t volume_group_rec_bytes(const VolGeo& g, int tz) {
    return sizeof(VolRec) * 32 * VG_WARPS * (size_t)tz * volume_tiles_plane(g);
}

cudaError_t launch_volume_plane(const VolPlaneArgs& a, int nz, const VolFilterArgs* f, int most, cudaStream_t s) {
    dim3 grid((a.W - VE + VP_NX) / VP_NX, (a.H - VE + VP_NY) / VP_NY, nz);
    const int per = grid.x * grid.y, zs = f ? (VS_GROUPS + per - 1) / per : 0;
    grid.z += zs;
    if (!f) volume_plane_kernel<0><<<grid, 128, 0, s>>>(a, VolFilterArgs{}, zs, 0);
    else if (f->g.K == 32) volume_plane_kernel<32><<<grid, 128, 0, s>>>(a, *f, zs, most);
    else if (f->g.K == 16) volume_plane_kernel<16><<<grid, 128, 0, s>>>(a, *f, zs, most);
    else return cudaErrorInvalidValue;
    return cudaGetLastError();
}

cudaError_t launch_volume_group(const VolGroupArgs& a, int tz, cudaStream_t s) {
    const int tiles = tz * volume_tiles_plane(a.f.g);
    switch (a.f.g.K) {
        case 2: return launch_vg<2>(a, tiles, s);
        case 4: return launch_vg<4>(a, tiles, s);
        case 8: return launch_vg<8>(a, tiles, s);
        case 16: return launch_vg<16>(a, tiles, s);
        case 32: return launch_vg<32>(a, tiles, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace htsvd
