// Dispatch of the group filter on projection planes.
#include <algorithm>
#include <type_traits>

#include "group_impl.cuh"
#include "sample_rows.cuh"

namespace htsvd {

namespace {

template <int K, int C, typename Tin, bool MF, bool ADJ = false>
cudaError_t launch_group_t(const GroupArgs& a, int grid, cudaStream_t s) {
    const int smem = group_layout<C>(a.f.FHmax, a.f.FWmax, a.cap, ADJ).total;
    auto fn = group_kernel<K, C, Tin, MF, ADJ>;
    cudaError_t e = allow_smem(fn, 64);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    fn<<<grid, GR_THREADS, smem, s>>>(a);
    return cudaGetLastError();
}

template <int K, int C>
cudaError_t dispatch(const GroupArgs& a, int grid, cudaStream_t s) {
    if (a.f.mode == FM_ADJOINT)
        return a.f.img_is_float ? launch_group_t<K, C, float, false, true>(a, grid, s) : cudaErrorInvalidValue;
    if (a.f.mode == FM_VIDEO) return a.f.img_is_float ? cudaErrorInvalidValue : launch_group_t<K, C, uint8_t, true>(a, grid, s);
    return a.f.img_is_float ? launch_group_t<K, C, float, false>(a, grid, s)
                            : launch_group_t<K, C, uint8_t, false>(a, grid, s);
}

template <int C>
cudaError_t dispatch_k(const GroupArgs& a, int grid, cudaStream_t s) {
    switch (a.f.g.K) {
        case 2: return dispatch<2, C>(a, grid, s);
        case 4: return dispatch<4, C>(a, grid, s);
        case 8: return dispatch<8, C>(a, grid, s);
        case 16: return dispatch<16, C>(a, grid, s);
        case 32: return dispatch<32, C>(a, grid, s);
    }
    return cudaErrorInvalidValue;
}

GLayout layout_of(const GroupArgs& a, int cap) {
    const bool adj = a.f.mode == FM_ADJOINT;
    return a.f.g.C == 3 ? group_layout<3>(a.f.FHmax, a.f.FWmax, cap, adj)
                        : group_layout<1>(a.f.FHmax, a.f.FWmax, cap, adj);
}

template <int K, int C, typename Tin, bool MF>
__global__ void __launch_bounds__(K * PS) sample_rows_kernel(FilterArgs a, int* __restrict__ st, int most) {
    __shared__ float sm[K * PS2 * C];
    __shared__ unsigned mask[PS];
    sample_group<K, C, Tin, MF, K * PS>(a, blockIdx.x, sm, mask, st, most);
}

template <int K>
cudaError_t sample_rows(const FilterArgs& a, int most, int* st, cudaStream_t s) {
    const bool mf = a.mode == FM_VIDEO;
    most *= SR_GROUPS;
    if (a.g.C == 3) {
        if (mf) sample_rows_kernel<K, 3, uint8_t, true><<<SR_GROUPS, K * PS, 0, s>>>(a, st, most);
        else if (a.img_is_float) sample_rows_kernel<K, 3, float, false><<<SR_GROUPS, K * PS, 0, s>>>(a, st, most);
        else sample_rows_kernel<K, 3, uint8_t, false><<<SR_GROUPS, K * PS, 0, s>>>(a, st, most);
    } else {
        if (mf) sample_rows_kernel<K, 1, uint8_t, true><<<SR_GROUPS, K * PS, 0, s>>>(a, st, most);
        else if (a.img_is_float) sample_rows_kernel<K, 1, float, false><<<SR_GROUPS, K * PS, 0, s>>>(a, st, most);
        else sample_rows_kernel<K, 1, uint8_t, false><<<SR_GROUPS, K * PS, 0, s>>>(a, st, most);
    }
    return cudaGetLastError();
}

// Denominator sum_g w_g (patches covering a pixel) of a tile of references: the weights are added at the
// patches' origins (the K positions of a group are distinct, one lane each, groups in order: a fixed order of
// sums), and every pixel takes the 8 x 8 box sum of the origins that reach it. Partials as the group
// filter's for one channel, (0, denominator). 32 adds per group in place of 2,048 weights.
constexpr int DN_THREADS = 128;

__global__ void __launch_bounds__(DN_THREADS) denom_kernel(const __grid_constant__ FilterArgs a, int* __restrict__ st) {
    extern __shared__ float dsm[];
    const int tile = blockIdx.x;
    if (st && tile == 0 && threadIdx.x < 3) st[threadIdx.x] = 0;
    const Geo& g = a.g;
    const int tid = threadIdx.x, ty = tile / a.ntx, tx = tile - ty * a.ntx;
    int FY0, FY1, FX0, FX1;
    tile_span(ty, a.TR, g.nry, g.s, g.H, g.npy, g.wny, g.win, FY0, FY1);
    tile_span(tx, a.TR, g.nrx, g.s, g.W, g.npx, g.wnx, g.win, FX0, FX1);
    const int FH = FY1 - FY0, FW = FX1 - FX0, OH = FH - PS + 1, OW = FW - PS + 1;
    float* org = dsm;                                  // [OH][OW]
    float* row = dsm + a.FHmax * a.FWmax;              // [OH][FW]: sums of 8 origins along x
    for (int t = tid; t < OH * OW; t += DN_THREADS) org[t] = 0.f;
    __syncthreads();
    if (tid < 32) {
        const int iy0 = ty * a.TR, ix0 = tx * a.TR;
        const int th = min(a.TR, g.nry - iy0), tw = min(a.TR, g.nrx - ix0);
        for (int q = 0; q < th * tw; ++q) {
            const int grp = (iy0 + q / tw) * g.nrx + ix0 + q % tw;
            const float w = a.w_in ? a.w_in[grp] : 1.f;
            if (tid < g.K) {
                // (a caller-given index outside the footprint is clamped into it; two lanes may then meet)
                const int v = a.idx[(size_t)grp * g.K + tid];
                const int y = v / g.W, x = v - y * g.W;
                const int oy = min(max(y - FY0, 0), OH - 1), ox = min(max(x - FX0, 0), OW - 1);
                atomicAdd(org + oy * OW + ox, w);
            }
            __syncwarp();
        }
    }
    __syncthreads();
    for (int t = tid; t < OH * FW; t += DN_THREADS) {
        const int y = t / FW, x = t - y * FW;
        float s = 0.f;
        for (int j = max(0, x - OW + 1); j < PS && j <= x; ++j) s += org[y * OW + x - j];
        row[t] = s;
    }
    __syncthreads();
    float2* dst = reinterpret_cast<float2*>(a.partials) + (size_t)tile * a.FHmax * a.FWmax;
    for (int t = tid; t < FH * FW; t += DN_THREADS) {
        const int y = t / FW, x = t - y * FW;
        float s = 0.f;
        for (int i = max(0, y - OH + 1); i < PS && i <= y; ++i) s += row[(y - i) * FW + x];
        dst[y * a.FWmax + x] = make_float2(0.f, s);
    }
}

// dot[position] = <patch of u, patch of v> over the image (8 x 8 box sums of the channels' products), rows
// py0 .. py0 + rows - 1 of positions.
constexpr int DP_X = 64, DP_Y = 16;

__global__ void __launch_bounds__(256) patch_dot_kernel(const float* __restrict__ u, const float* __restrict__ v, int H,
                                                        int W, int C, int py0, int rows, float* __restrict__ dot) {
    __shared__ float e[DP_Y + PS - 1][DP_X + PS], hs[DP_Y + PS - 1][DP_X];
    const int x0 = blockIdx.x * DP_X, r0 = blockIdx.y * DP_Y, y0 = py0 + r0, tid = threadIdx.x;
    for (int t = tid; t < (DP_Y + PS - 1) * (DP_X + PS - 1); t += 256) {
        const int r = t / (DP_X + PS - 1), c = t - r * (DP_X + PS - 1);
        float s = 0.f;
        if (y0 + r < H && x0 + c < W) {
            const size_t p = ((size_t)(y0 + r) * W + x0 + c) * C;
            for (int k = 0; k < C; ++k) s = fmaf(u[p + k], v[p + k], s);
        }
        e[r][c] = s;
    }
    __syncthreads();
    for (int t = tid; t < (DP_Y + PS - 1) * DP_X; t += 256) {
        const int r = t / DP_X, c = t - r * DP_X;
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < PS; ++j) s += e[r][c + j];
        hs[r][c] = s;
    }
    __syncthreads();
    for (int t = tid; t < DP_Y * DP_X; t += 256) {
        const int r = t / DP_X, c = t - r * DP_X;
        if (r0 + r >= rows || x0 + c > W - PS) continue;
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < PS; ++i) s += hs[r + i][c];
        dot[(size_t)(r0 + r) * (W - PS + 1) + x0 + c] = s;
    }
}

}  // namespace

// Where planes and group filter take as long as the tile kernel alone. The fewer groups a tile holds, the fewer warps
// work on it (with one, a third of them), and the earlier that is. us of both, stride 3, window 18, by the mean rows,
// on pictures at the universal threshold (tile edge, references): RGB, K 32: 1, 4,030: 171 / 176 at 19, 196 / 180 at
// 32; 1, 7,308: 271 / 307 at 17, 323 / 315 at 31; 2, 10,395: 267 / 292 at 30, 348 / 306 at 47; 2, 16,854: 397 / 464 at
// 30, 488 / 484 at 46; 3, 31,265: 786 / 805 at 45, 880 / 819 at 63; 4, 52,735: 1,147 / 1,293 at 45, 1,517 / 1,316 at 63.
// Gray, K 32: 1, 7,308: 186 / 204 at 21, 242 / 213 at 46; 2, 10,395: 151 / 168 at 20, 203 / 174 at 41; 3, 22,499: 318 /
// 317 at 39. RGB, K 16: 1, 4,030: 137 / 155 at 24, 160 / 161 at 39; more: 221 / 250 at 39 (10,395). Gray, K 16: 1,
// 4,030: 97 / 103 at 19, 113 / 104 at 32; 2, 10,395: 119 / 131 at 20, 140 / 133 at 31. At lower thresholds, where every
// group keeps a few coefficients in most of its slots, the lines lie a third lower (RGB, K 32, 3 x 3: 763 / 750 at 34),
// and the sample's 15 us count in smaller images: the limits lie between. With 8 slots or fewer the group filter is
// the faster one at any threshold.
//
// The backward pass: RGB, K 32: one group a tile, 4,030 references, ratio of the tile kernel's time 1.05 at 19, 0.99 at 32;
// 7,308: 1.08 at 31, 0.95 at 48; more groups: 1.23 at 63, 0.95 at 77. Gray, K 32: one group, 4,030: 1.12 at 22, 0.83 at
// 43; 7,308: 1.23 at 21, 0.98 at 46; more: 1.26 at 70, 0.84 at 158. RGB, K 16: one group, 4,030: 1.06 at 15, 1.00 at 24;
// 7,308: 1.06 at 30, 1.00 at 38; more: 1.01 at 84. Gray, K 16: one group, 4,030: 0.98 at 8; 7,308: 1.11 at 9, 1.00 at 18;
// more: 1.04 at 77. K 8: at any, but for small gray images (K 2, 4,225 references: 0.89). Below 3,000 references (K 32:
// 1,500; us: 961 139 / 96 at 5, 1,681 135 / 149 at 5, 344 / 276 at 245; K 16, 1,681 101 / 88 at 3) the tile kernel, but
// for images of so few references that its tiles are the largest and fewer than the SMs (289: 344 / 580 at 5, 225:
// 1,143 / 1,085 at 173).
int group_rows_limit(const FilterArgs& a) {
    const int K = a.g.K, ng = a.g.ngroups();
    const bool rgb = a.g.C == 3;
    if (a.mode == FM_ADJOINT) {
        if (ng < (K == 32 ? 1500 : 3000)) {
            if (a.ntx * a.nty >= device_sm_count()) return -1;
            return K == 32 ? 60 : K == 16 ? 40 : kEveryRow;
        }
        if (K <= 8) return !rgb && ng < 5000 ? -1 : kEveryRow;
        if (K == 32 && ng < 4000) return 14;
        if (a.TR > 1) return rgb ? (K == 32 ? 72 : 84) : K == 32 ? 110 : 100;
        if (K == 32) return ng < 5000 ? 24 : rgb ? 32 : 36;
        return rgb ? (ng < 4000 ? 9 : ng < 5000 ? 17 : 28) : ng < 4000 ? 3 : ng < 5000 ? 7 : 16;
    }
    if (K <= 8) return kEveryRow;
    if (ng < 5000) return (rgb ? (K == 32 ? 20 : 30) : 18) * (ng < 4000 ? 2 : 3) / 3;
    constexpr int rgb32[] = {26, 32, 38, 40, 42}, gray32[] = {24, 28, 32, 34, 36};
    constexpr int rgb16[] = {36, 40, 48, 48, 48}, gray16[] = {26, 28, 36, 40, 48};
    const int t = std::min(a.TR, 5) - 1;
    return K == 32 ? (rgb ? rgb32 : gray32)[t] : (rgb ? rgb16 : gray16)[t];
}

cudaError_t launch_sample_rows(const FilterArgs& a, int most, int* st, cudaStream_t s) {
    return a.g.K == 32   ? sample_rows<32>(a, most, st, s)
           : a.g.K == 16 ? sample_rows<16>(a, most, st, s)
                         : cudaErrorInvalidValue;
}

cudaError_t launch_denom(const FilterArgs& a, int* st, cudaStream_t s) {
    const size_t smem = 2 * sizeof(float) * a.FHmax * a.FWmax;
    cudaError_t e = allow_smem(denom_kernel);
    if (e != cudaSuccess) return e;
    denom_kernel<<<a.ntx * a.nty, DN_THREADS, smem, s>>>(a, st);
    return cudaGetLastError();
}

cudaError_t launch_patch_dot(const float* u, const float* v, int H, int W, int C, int py0, int rows, float* dot,
                             cudaStream_t s) {
    patch_dot_kernel<<<dim3((W - PS + DP_X) / DP_X, (rows + DP_Y - 1) / DP_Y), 256, 0, s>>>(u, v, H, W, C, py0, rows, dot);
    return cudaGetLastError();
}

int group_grid(GroupArgs& a) {
    // as many CTAs per SM as the registers allow and whose accumulators leave room for the row lists
    const int rows = a.f.g.K * PS;                        // every row of every slot
    const int row_bytes = GR_WARPS * PS * a.f.g.C * 4;     // all warps
    const int fixed = layout_of(a, 0).total + 1024 + 64;
    a.per_sm = 1;
    a.cap = std::min(rows, 8);
    for (int n = GR_CTAS; n >= 1; --n) {
        const int room = 228 * 1024 / n - fixed;
        const int cap = std::min(rows, room / row_bytes);
        if (cap >= std::min(rows, 16) || n == 1) {
            a.per_sm = n;
            a.cap = std::max(cap, 0);
            break;
        }
    }
    // Candidate rows of a first step from which a tile is left to filter_tile_fwd. us per 512 x 512 RGB image, K 32,
    // stride 3, for limits 12 / 18 / 24 / 30 / 38: 973 / 897 / 908 / 842 / 838 at sigma 25 and multiplier 3.2,
    // 860 / 816 / 762 / 764 / 763 at sigma 15 and 4.2, 1,483 / 1,489 / 1,479 / 1,781 / 1,860 at sigma 8 and 2.0. With
    // 8 patches or fewer a group has 64 rows at most and nothing is left.
    a.dense_rows = a.f.g.K <= 8 ? 1 << 20 : 30;
    return std::min(a.nty_band * a.f.ntx, a.per_sm * device_sm_count());
}

size_t group_spill_floats(const GroupArgs& a, int grid) {
    return (size_t)grid * GR_WARPS * group_spill_warp(a.f.g.K, a.f.g.C);
}

cudaError_t launch_group(const GroupArgs& args, int grid, cudaStream_t s) {
    GroupArgs a = args;
    a.wrec = (unsigned)(((unsigned long long)1 << 32) / (unsigned)a.f.g.W);
    return a.f.g.C == 3 ? dispatch_k<3>(a, grid, s) : dispatch_k<1>(a, grid, s);
}

}  // namespace htsvd
