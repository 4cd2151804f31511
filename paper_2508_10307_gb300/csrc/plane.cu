// Projection planes: the t-SVD projection S = U^T * P * V (Eq. (forward transform)) of the patch at
// every position of a band of image rows, written once to HBM and gathered by the group filter.
//
// A position belongs to K / stride^2 groups on average (3.6 at K 32, stride 3), and neighbouring
// patches share their column transforms, so projecting each position once costs 2,880 FMA against
// 5,120 FMA per group member inside the filter.
//
// One CTA (4 warps) takes PL_NX x 8 positions. Stage A: thread (column x, every second row) forms
// Y_f[i](y, x) = sum_a conj(U_f[a][i]) X_f(y + a, x) for the 8 basis rows into shared memory, two basis
// rows (i, i + 4) per packed FMA. Stage B: warp = position row, lane = (basis row i < 4, basis column
// j): S_f[i][j](y, x) = sum_b Y_f[i](y, x + b) V_f[b][j] for the rows i and i + 4 as one packed pair,
// the eight Y columns in a register window that slides along x (two shared loads per position), the
// inverse channel DFT, and coalesced stores. Every sum keeps the term order of the
// filter's own projection stages (filter_impl.cuh), so both give the same coefficients bit for bit.
// Layout of a position, lane l = basis row l / 8 of a half h (rows 4 h ..), basis column l % 8: C = 3:
// per half, channels 0 and 1 of lane l at 2 l, 2 l + 1, then channel 2 at 64 + l; C = 1: halves 0 and 1 of
// lane l at 2 l, 2 l + 1.
#include "f32x2.cuh"
#include "kernels.h"
#include "sample_rows.cuh"

namespace htsvd {

namespace {

constexpr int PL_NX = 57;                    // positions per CTA row (64 columns staged)
constexpr int PL_COLS = PL_NX + PS - 1;
constexpr int PL_NY = 8;
constexpr int PL_THREADS = 128;
constexpr float P_S3H = 0.866025403784438646763723170752936183f;   // sqrt(3)/2
constexpr float P_SQ3 = 1.73205080756887729352744634150587237f;    // sqrt(3)
constexpr float P_THIRD = 0.333333333333333333333333333333333333f;

template <int C>
struct PCfg {
    static constexpr int UPF = (C == 3) ? 8 : 2;     // floats per (a, i) of the paired U table
    static constexpr int YF = (C == 3) ? 8 : 2;      // floats per (y, x, i) of the paired Y buffer
    static constexpr int U_BYTES = PS * 4 * UPF * 4;
    static constexpr int Y_BYTES = PL_NY * PL_COLS * 4 * YF * 4;
    static constexpr int Q_BYTES = PL_NY * PL_COLS * 4;
};

template <int C, typename Tin>
__host__ __device__ constexpr int plane_smem() {
    return PCfg<C>::U_BYTES + PCfg<C>::Y_BYTES + PCfg<C>::Q_BYTES + (PL_NY + PS - 1) * PL_COLS * C * (int)sizeof(Tin);
}

// SK: slots of the groups that the first zs slices of blocks sample (0: no such slices).
template <int C, typename Tin, int SK>
__global__ void __launch_bounds__(PL_THREADS, 3) plane_kernel(const __grid_constant__ PlaneArgs a,
                                                              const __grid_constant__ FilterArgs f, int zs, int most,
                                                              int* __restrict__ st) {
    using P = PCfg<C>;
    extern __shared__ __align__(16) unsigned char sm[];
    if constexpr (SK > 0) {
        __shared__ unsigned mask[PS];
        if ((int)blockIdx.z < zs) {
            const int b = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
            if (b < SR_GROUPS)
                sample_group<SK, C, Tin, false, PL_THREADS>(f, b, reinterpret_cast<float*>(sm), mask, st, most);
            return;
        }
    }
    float* ut = reinterpret_cast<float*>(sm);
    float* yb = reinterpret_cast<float*>(sm + P::U_BYTES);
    float* qs = reinterpret_cast<float*>(sm + P::U_BYTES + P::Y_BYTES);
    Tin* px = reinterpret_cast<Tin*>(sm + P::U_BYTES + P::Y_BYTES + P::Q_BYTES);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int npx = a.W - PS + 1;
    const int x0 = blockIdx.x * PL_NX, yr0 = blockIdx.y * PL_NY;       // yr0: row within the band
    const int y0 = a.py0 + yr0;
    const Tin* img = reinterpret_cast<const Tin*>(a.img);
    if (a.counter && blockIdx.x == 0 && blockIdx.y == 0 && (int)blockIdx.z == zs && tid < 2) a.counter[tid] = 0;
    if constexpr (SK > 0) {                            // (by now known to be dense: nobody reads the planes)
        if (__syncthreads_or(tid == 0 && *(volatile const int*)a.dense)) return;
    } else {
        if (a.dense && *a.dense) return;
    }

    for (int t = tid; t < PS * 4; t += PL_THREADS) {
        const int r = t >> 2, i = t & 3;
        float* d = ut + t * P::UPF;
        d[0] = a.basis32[r * PS + i];
        d[1] = a.basis32[r * PS + i + 4];
        if constexpr (C == 3) {
            d[2] = a.basis32[64 + r * PS + i];
            d[3] = a.basis32[64 + r * PS + i + 4];
            d[4] = a.basis32[128 + r * PS + i];
            d[5] = a.basis32[128 + r * PS + i + 4];
            d[6] = -d[4];
            d[7] = -d[5];
        }
    }
    const int rows = min(PL_NY + PS - 1, a.H - y0), cols = min(PL_COLS, a.W - x0);
    for (int t = tid; t < (PL_NY + PS - 1) * PL_COLS * C; t += PL_THREADS) {
        const int r = t / (PL_COLS * C), c = t - r * (PL_COLS * C);
        px[t] = (r < rows && c < cols * C) ? img[((size_t)(y0 + r) * a.W + x0) * C + c] : (Tin)0;
    }
    __syncthreads();

    // ---- stage A: column x, rows yq, yq + 2, ...
    {
        const int x = tid & 63, yq = tid >> 6;
#pragma unroll 1
        for (int y = yq; y < PL_NY; y += PL_THREADS / 64) {
            const Tin* src = px + (y * PL_COLS + x) * C;
            float q = 0.f;
            f2 s0[4], sr[4], si[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) s0[i] = sr[i] = si[i] = f2_dup(0.f);
#pragma unroll 2
            for (int r = 0; r < PS; ++r) {
                if constexpr (C == 3) {
                    const float v0 = (float)src[r * PL_COLS * 3], v1 = (float)src[r * PL_COLS * 3 + 1],
                                v2 = (float)src[r * PL_COLS * 3 + 2];
                    q = fmaf(v0, v0, q);
                    q = fmaf(v1, v1, q);
                    q = fmaf(v2, v2, q);
                    const f2 X0 = f2_dup(v0 + v1 + v2);
                    const f2 Xr = f2_dup(v0 - 0.5f * (v1 + v2));
                    const f2 Xi = f2_dup(P_S3H * (v2 - v1));
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const ulonglong2 u01 = *reinterpret_cast<const ulonglong2*>(ut + (r * 4 + i) * 8);
                        const ulonglong2 u23 = *reinterpret_cast<const ulonglong2*>(ut + (r * 4 + i) * 8 + 4);
                        s0[i] = f2_fma(u01.x, X0, s0[i]);
                        sr[i] = f2_fma(u01.y, Xr, f2_fma(u23.x, Xi, sr[i]));
                        si[i] = f2_fma(u01.y, Xi, f2_fma(u23.y, Xr, si[i]));
                    }
                } else {
                    const float v0 = (float)src[r * PL_COLS];
                    q = fmaf(v0, v0, q);
                    const f2 X0 = f2_dup(v0);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        s0[i] = f2_fma(*reinterpret_cast<const f2*>(ut + (r * 4 + i) * 2), X0, s0[i]);
                }
            }
            qs[y * PL_COLS + x] = q;
            float* d = yb + (size_t)(y * PL_COLS + x) * 4 * P::YF;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if constexpr (C == 3) {
                    *reinterpret_cast<ulonglong2*>(d + i * 8) = make_ulonglong2(s0[i], sr[i]);
                    *reinterpret_cast<f2*>(d + i * 8 + 4) = si[i];
                } else {
                    *reinterpret_cast<f2*>(d + i * 2) = s0[i];
                }
            }
        }
    }
    __syncthreads();

    const int nx = min(PL_NX, npx - x0), ny = min(PL_NY, a.rows - yr0);
    // squared norm of each patch: eight column sums
    for (int t = tid; t < ny * PL_NX; t += PL_THREADS) {
        const int y = t / PL_NX, x = t - y * PL_NX;
        if (x < nx) {
            const float* q = qs + y * PL_COLS + x;
            float s = 0.f;
#pragma unroll
            for (int b = 0; b < PS; ++b) s += q[b];
            a.pn[(size_t)(yr0 + y) * npx + x0 + x] = s;
        }
    }

    // ---- stage B: position rows warp, warp + 4; lane = (basis row il, basis column j)
    const int il = lane >> 3, j = lane & 7;
    if constexpr (C == 3) {
        f2 v0[PS], vr[PS], vi[PS], nv[PS];
#pragma unroll
        for (int b = 0; b < PS; ++b) {
            v0[b] = f2_dup(a.basis32[192 + b * PS + j]);
            vr[b] = f2_dup(a.basis32[256 + b * PS + j]);
            vi[b] = f2_dup(a.basis32[320 + b * PS + j]);
            nv[b] = f2_dup(-a.basis32[320 + b * PS + j]);
        }
#pragma unroll 1
        for (int row = warp; row < ny; row += PL_THREADS / 32) {
        const float* yrow = yb + (size_t)(row * PL_COLS) * 4 * P::YF + il * P::YF;
        float* dst = a.coef + ((size_t)(yr0 + row) * npx + x0) * (PS2 * C) + lane * 2;
        f2 w0[PS], wr[PS], wi[PS];                   // Y columns x .. x + 7, slot = column mod 8
        auto fetch = [&](int x, int slot) {
            const ulonglong2 p = *reinterpret_cast<const ulonglong2*>(yrow + x * 32);
            w0[slot] = p.x;
            wr[slot] = p.y;
            wi[slot] = *reinterpret_cast<const f2*>(yrow + x * 32 + 4);
        };
#pragma unroll
        for (int b = 0; b < PS - 1; ++b) fetch(b, b);
        const f2 two = f2_dup(2.f), third = f2_dup(P_THIRD), sq3 = f2_dup(P_SQ3), nsq3 = f2_dup(-P_SQ3);
#pragma unroll 1
        for (int xb = 0; xb < nx; xb += PS) {
#pragma unroll
            for (int u = 0; u < PS; ++u) {
                const int x = xb + u;
                if (x < nx) {                        // warp-uniform
                    fetch(x + PS - 1, (u + PS - 1) & 7);
                    f2 s0 = f2_dup(0.f), sr = s0, si = s0;
#pragma unroll
                    for (int b = 0; b < PS; ++b) {
                        const int k = (u + b) & 7;
                        s0 = f2_fma(w0[k], v0[b], s0);
                        sr = f2_fma(wr[k], vr[b], f2_fma(wi[k], nv[b], sr));
                        si = f2_fma(wr[k], vi[b], f2_fma(wi[k], vr[b], si));
                    }
                    const f2 d01 = f2_sub(s0, sr);
                    const f2 o0 = f2_mul(f2_fma(two, sr, s0), third);
                    const f2 o1 = f2_mul(f2_fma(nsq3, si, d01), third);
                    const f2 o2 = f2_mul(f2_fma(sq3, si, d01), third);
                    float* o = dst + (size_t)x * 192;
                    float lo0, hi0, lo1, hi1;
                    f2_unpack(o0, lo0, hi0);
                    f2_unpack(o1, lo1, hi1);
                    *reinterpret_cast<f2*>(o) = f2_pack(lo0, lo1);
                    *reinterpret_cast<f2*>(o + 96) = f2_pack(hi0, hi1);
                    f2_unpack(o2, lo0, hi0);
                    o[64 - lane] = lo0;
                    o[160 - lane] = hi0;
                }
            }
        }
        }
    } else {
        f2 v0[PS], w0[PS];
#pragma unroll
        for (int b = 0; b < PS; ++b) v0[b] = f2_dup(a.basis32[64 + b * PS + j]);
#pragma unroll 1
        for (int row = warp; row < ny; row += PL_THREADS / 32) {
        const float* yrow = yb + (size_t)(row * PL_COLS) * 4 * P::YF + il * P::YF;
        float* dst = a.coef + ((size_t)(yr0 + row) * npx + x0) * (PS2 * C) + lane * 2;
#pragma unroll
        for (int b = 0; b < PS - 1; ++b) w0[b] = *reinterpret_cast<const f2*>(yrow + b * 8);
#pragma unroll 1
        for (int xb = 0; xb < nx; xb += PS) {
#pragma unroll
            for (int u = 0; u < PS; ++u) {
                const int x = xb + u;
                if (x < nx) {
                    w0[(u + PS - 1) & 7] = *reinterpret_cast<const f2*>(yrow + (x + PS - 1) * 8);
                    f2 s0 = f2_dup(0.f);
#pragma unroll
                    for (int b = 0; b < PS; ++b) s0 = f2_fma(w0[(u + b) & 7], v0[b], s0);
                    *reinterpret_cast<f2*>(dst + (size_t)x * 64) = s0;
                }
            }
        }
        }
    }
}

template <int C, typename Tin, int SK = 0>
cudaError_t launch_plane_t(const PlaneArgs& a, cudaStream_t s, const FilterArgs* f = nullptr, int most = 0,
                           int* st = nullptr) {
    constexpr int smem = plane_smem<C, Tin>();
    static_assert(smem >= SK * PS2 * C * 4, "the sample's patches");
    auto fn = plane_kernel<C, Tin, SK>;
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    dim3 grid((a.W - PS + PL_NX) / PL_NX, (a.rows + PL_NY - 1) / PL_NY);
    const int per = grid.x * grid.y, zs = SK > 0 ? (SR_GROUPS + per - 1) / per : 0;
    grid.z = zs + 1;
    fn<<<grid, PL_THREADS, smem, s>>>(a, f ? *f : FilterArgs{}, zs, most * SR_GROUPS, st);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_plane(const PlaneArgs& a, cudaStream_t s, const FilterArgs* f, int most, int* st) {
    if (f) {
        if (!a.is_float || !a.dense || (f->g.K != 32 && f->g.K != 16)) return cudaErrorInvalidValue;
        if (f->g.K == 32)
            return a.C == 3 ? launch_plane_t<3, float, 32>(a, s, f, most, st) : launch_plane_t<1, float, 32>(a, s, f, most, st);
        return a.C == 3 ? launch_plane_t<3, float, 16>(a, s, f, most, st) : launch_plane_t<1, float, 16>(a, s, f, most, st);
    }
    if (a.C == 3) return a.is_float ? launch_plane_t<3, float>(a, s) : launch_plane_t<3, uint8_t>(a, s);
    return a.is_float ? launch_plane_t<1, float>(a, s) : launch_plane_t<1, uint8_t>(a, s);
}

}  // namespace htsvd
