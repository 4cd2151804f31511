// Internal launch interface between the C-ABI layer (api.cu) and the kernels.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include "common.cuh"

namespace htsvd {

enum MatchMode { MM_GRAY = 0, MM_GCP = 1, MM_FULL = 2, MM_GREEN = 3 };

// Streaming multiprocessors of the calling thread's current device (cudaDevAttrMultiProcessorCount,
// looked up once per device); grids and wave counts are sized from it.
int device_sm_count();

// Lets launches of fn take dynamic shared memory up to what a CTA can have beside `fixed` bytes of static. The same
// limit whatever a launch needs: a smaller one set by another host thread, between this request and the launch
// that needs more, would make that launch fail.
constexpr int kSmemOptIn = 227 * 1024;
template <typename F>
cudaError_t allow_smem(F* fn, int fixed = 0) {
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemOptIn - fixed);
}

// ---- block matching (bm.cu)
struct BMArgs {
    const uint8_t* img;
    Geo g;
    int mode;            // MatchMode (resolved: gray for C = 1)
    double gamma2;       // gcp_gamma^2
    int rstep;           // reference subsampling (1 = every reference)
    int nry_s, nrx_s;    // references per axis after subsampling
    int TRy, TRx;        // references per tile
    int32_t* idx;        // out [nry_s * nrx_s][K]
    // Spatio-temporal search (video): candidates also come from frames f0 .. f0 + nfr - 1 of the
    // clip at vid (frame stride fstride bytes); img is frame fref. Indices are global,
    // f * H * W + y * W + x. nfr = 0 (the default) searches img alone, with frame-local indices.
    const uint8_t* vid;
    long long fstride;
    int f0, nfr, fref;
};
size_t bm_smem_bytes(const BMArgs& a);
// Halves the tile (TRx, TRy) until its shared-memory footprint leaves room for two CTAs per SM.
void bm_fit_tiles(BMArgs& a);
cudaError_t launch_block_match(const BMArgs& a, cudaStream_t s);
// Tensor-core form: bytes of device scratch it needs (0: not for this geometry, or not faster there), and
// its launch. timeout: host-readable word set if a wait inside the kernel runs out (give_up: as if one had); the
// groups then hold positions of the search windows that may not be the nearest.
size_t bm_tc_scratch(const BMArgs& a, int share);
cudaError_t launch_block_match_tc(const BMArgs& a, void* scratch, int* timeout, bool give_up, cudaStream_t s);

// ---- second moments and bases (moments.cu)
// Row/column second moments of the reference patches, exact:
//   R[a][a'][c][c'] = sum_r sum_b P_r[a][b][c] P_r[a'][b][c']
//   Q[b][b'][c][c'] = sum_r sum_a P_r[a][b][c] P_r[a][b'][c']
// stored as uint64 [2][8][8][C][C] (R then Q).
cudaError_t launch_moments(const uint8_t* img, const Geo& g, unsigned long long* d_mom, cudaStream_t s);
// Row and column moments derived exactly from the full second moment (lower triangle) that
// launch_full_moment wrote; replaces launch_moments where the full moment is already formed.
cudaError_t launch_moments_from_full(const unsigned long long* d_M, int C, unsigned long long* d_mom, cudaStream_t s);
// Full second moment M[u][v] = sum_r p_r[u] p_r[v] (d = 64 C) and s[u] = sum_r p_r[u], uint64.
cudaError_t launch_full_moment(const uint8_t* img, const Geo& g, unsigned long long* d_M,
                               unsigned long long* d_s, cudaStream_t s);
// FP64 eigen-solve of the per-slice row/column scatter matrices -> canonical bases.
//   basis64: [2 (U,V)][C][8][8] complex (re, im), slice f, row a, column i.
//   basis32: packed float slices for the filter (U0r, [U1r, U1i], V0r, [V1r, V1i]), each [a][i].
//   gap (optional): per solved problem (U slices f = 0 .. C/2, then V slices; basis_problems(C) of them)
//   the smallest gap between consecutive eigenvalues relative to the largest eigenvalue.
inline int basis_problems(int C) { return 2 * (C / 2 + 1); }
cudaError_t launch_basis(const unsigned long long* d_mom, int C, double* d_basis64, float* d_basis32,
                         cudaStream_t s, double* d_gap = nullptr);
// Row and column moments (layout as launch_moments) of a cube with any number of bands g.C.
cudaError_t launch_cube_moments(const uint8_t* img, const Geo& g, unsigned long long* d_mom, cudaStream_t s);
// Floats of the packed FP32 basis: C in {1, 3}: 512 (the filter's layout); cubes (other C):
// [2 (U, V)][C/2 + 1 slices][re, im][8][8].
inline int basis32_floats(int C) { return (C == 1 || C == 3) ? 512 : 2 * (C / 2 + 1) * 2 * 64; }
// Quantise a float image: q = clip(rint(x), 0, 255).
cudaError_t launch_quantize(const float* x, int64_t n, uint8_t* q, cudaStream_t s);

// ---- projection planes (plane.cu): the projected patch at every position of the image rows
// py0 .. py0 + rows - 1 (positions), 64 C floats each in the group filter's lane order, and its
// squared norm. basis32: the packed FP32 bases of launch_basis.
struct PlaneArgs {
    const void* img;         // uint8 or float H x W x C
    int is_float;
    int H, W, C;
    int py0, rows;
    const float* basis32;
    float* coef;             // [rows][W - 7][64 C]
    float* pn;               // [rows][W - 7]
    int* counter;            // optional: two words zeroed (the group filter's counters)
    const int* dense;        // optional: nothing else is done where it is set
};
// With f (float images, K 16 or 32), the sample of launch_sample_rows as well, into three zeroed words at st.
struct FilterArgs;
cudaError_t launch_plane(const PlaneArgs& a, cudaStream_t s, const FilterArgs* f = nullptr, int most = 0, int* st = nullptr);

// ---- group filter and aggregation (filter.cu)
enum FilterMode { FM_FORWARD = 0, FM_ADJOINT = 2, FM_VIDEO = 3, FM_ANALYZE = 4, FM_SYNTH = 5 };

// Guard band of the threshold decision: a coefficient whose FP32 value lies within
// kBandRel * ||G||_F + kBandTau * tau of tau is decided again in FP64 (||G||_F: Frobenius
// norm of the group's inputs; kBandTau covers tau rounded to FP32).
constexpr float kBandRel = 1.9073486328125e-06f;      // 2^-19
constexpr double kBandTau = 2.384185791015625e-07;    // 2^-22
// Cubes: band relative to the norm of the Haar slot being thresholded (its FP32 coefficient error,
// measured on 31-band cubes: 2^-23 of that norm).
constexpr float kBandRelCube = 1.9073486328125e-06f;   // 2^-19
struct FilterArgs {
    const void* img;         // uint8 or float H x W x C (the values that are filtered)
    int img_is_float;
    Geo g;
    int TR, ntx, nty;        // references per tile edge, tiles per axis
    int FHmax, FWmax;        // partial-footprint strides
    const int32_t* idx;      // [N][K]
    const float* basis32;
    const double* basis64;
    float tau32;
    double tau64;
    float band_rel;          // guard band: |S| within band_rel*||G||_F + band_abs of tau -> FP64 decision
    float band_abs;
    const float* w_in;       // optional per-group weights
    int agg_mode;
    float* partials;         // [ntiles][FHmax][FWmax][C+1]
    uint32_t* mask_out;      // optional
    float* weights_out;      // optional
    float* coef_out;         // optional FP32 coefficients, K*64*C per group (accuracy checks)
    int mode;                // FilterMode
    // adjoint inputs
    const float* r_img;      // (gout / D) image that is filtered with the masks of img (FM_ADJOINT)
    const float* out_img;    // forward output (FM_ADJOINT, for the weight gradient)
    float* grad_w;           // FM_ADJOINT, per group
    // FM_VIDEO (forward over a clip, uint8): groups of frame fref may hold patches of frames
    // f0 .. f0 + nfr - 1 of vid (frame stride fstride elements, indices f * H * W + y * W + x);
    // only the patches of frame fref are aggregated. img is frame fref.
    const void* vid;
    long long fstride;
    int f0, nfr, fref;
    // Coefficient cache of the noisy groups (threshold sweeps): FM_ANALYZE writes, FM_SYNTH reads
    // the Haar-domain coefficients of every group ([N][K][64 C] floats, unnormalised Haar, slot
    // order of the in-place transform), the per-patch squared norms ([N][32]) and ||G||_F^2 ([N],
    // the filter's own integer or float-bit representation).
    float* cache_coef;
    float* cache_pn;
    int* cache_nrm;
    // Tiles to filter (optional, device): counter[1] of them from counter[2] on, as the group filter leaves them.
    const int* left;
    // Where dense points to a word that is set: all left_tiles tiles from left_first on (the group filter has done none).
    const int* dense;
    int left_first, left_tiles;
};
// Group filter on projection planes (group.cu): the tiles of tile rows ty0 .. ty0 + nty_band - 1, their
// groups' coefficients gathered from the planes (one per frame in reach, planestride positions apart)
// instead of projected in the CTA; same partials as launch_filter. FM_FORWARD and FM_VIDEO.
struct GroupArgs {
    FilterArgs f;
    const float* coef;
    const float* pn;
    long long planestride;   // positions per frame plane
    int py0;                 // image row of the planes' first position row
    int ty0, nty_band;
    int cap;                 // rows of kept coefficients a warp holds in shared memory
    int per_sm;              // CTAs that share an SM
    float* spill;            // rows beyond cap, group_spill_floats(...) in all
    const float* rcoef;      // adjoint: planes of r
    const float* dot;        // adjoint: per position, <patch of r, patch of the output>
    // [0] tile counter, [1] number of tiles left over, [2 ...] those tiles: [0] and [1] zero at launch. A tile is
    // left over (no partial written) where its first groups keep more than dense_rows rows.
    int* counter;
    int dense_rows;
    unsigned wrec;           // 2^32 / W, rounded down (filled by the launch)
};
// Mean rows of coefficients a group keeps up to which planes and group filter are the faster way; kEveryRow: at
// any, -1: at none.
constexpr int kEveryRow = 1 << 20;
int group_rows_limit(const FilterArgs& a);
// Sets st[2] where the sampled groups of the image keep more rows than most in the mean (st: three zeroed words);
// FilterArgs as for the filter.
cudaError_t launch_sample_rows(const FilterArgs& a, int most, int* st, cudaStream_t s);
// Fills a.cap and a.per_sm and returns the grid (persistent CTAs) of a launch.
int group_grid(GroupArgs& a);
size_t group_spill_floats(const GroupArgs& a, int grid);
cudaError_t launch_group(const GroupArgs& a, int grid, cudaStream_t s);

// Denominator partials of a tiling (two floats per footprint pixel, (0, sum of the covering patches' weights)). Zeroes
// the three words at st, if given.
cudaError_t launch_denom(const FilterArgs& a, int* st, cudaStream_t s);
// dot[position] = <patch of u, patch of v> of two float images, position rows py0 .. py0 + rows - 1.
cudaError_t launch_patch_dot(const float* u, const float* v, int H, int W, int C, int py0, int rows, float* dot,
                             cudaStream_t s);

size_t filter_smem_bytes(const FilterArgs& a);
cudaError_t launch_filter(const FilterArgs& a, cudaStream_t s);
// out[p] = sum_tiles num / sum_tiles den (deterministic tile order). If den_out is set, the
// denominator plane is written too; if num_only, out = sum num (no division).
cudaError_t launch_reduce(const float* partials, const Geo& g, int TR, int ntx, int nty, int FHmax, int FWmax,
                          float* out, float* den_out, int num_only, const float* den_in, cudaStream_t s);
// z = y + eps b over n floats, each operation rounded once (the finite-difference SURE's perturbed image).
cudaError_t launch_perturb(const float* y, const float* b, float eps, int64_t n, float* z, cudaStream_t s);
// SURE terms in FP64: res[0] = sum (out - x)^2, res[1] = sum b * g over n floats (deterministic
// two-level reduction; scratch: sure_scratch_doubles() doubles).
size_t sure_scratch_doubles();
// Weight tuning (SURE of the per-group weights): u = alpha (f - x) - beta b; acc += a;
// w <- w exp(-step g / max|g|) (scratch: one unsigned, for max|g|).
cudaError_t launch_sure_cotangent(const float* f, const float* x, const float* b, float alpha, float beta, int64_t n,
                                  float* u, cudaStream_t s);
cudaError_t launch_add(const float* a, float* acc, int64_t n, cudaStream_t s);
cudaError_t launch_eg_update(float* w, const float* g, int64_t n, float step, unsigned* scratch, cudaStream_t s);
cudaError_t launch_sure_terms(const float* out, const float* x, const float* b, const float* g, int64_t n,
                              double* scratch, double* res, cudaStream_t s);
// Adjoint helper: r = gout / den.
cudaError_t launch_div(const float* gout, const float* den, int64_t npix, int C, float* r, cudaStream_t s);

// ---- small images of a batch, one launch a phase (small_batch.cuh)
constexpr int kSmallImages = 128;        // images a launch describes at most (its parameter: 9 KB)
struct SmallImage {
    const uint8_t* in;
    float* out;
    int32_t* idx;
    double tau;
    long long part;          // first float of its tile partials
    int H, W;
    int TR, TRy, TRx;        // filter tile edge, grouping tile
    int mom0, bm0, flt0, red0;   // work items of the images before it, per phase
};
struct SmallBatch {
    int n, C, s, win, K, mode, agg_mode;
    int per;                 // references per chunk of the moments
    double gamma2;
    unsigned long long* mom; // [n][2][64][C][C], zeroed
    double* b64;             // [n][2][C][64][2]
    float* b32;              // [n][512]
    float* part;
    SmallImage im[kSmallImages];
};
cudaError_t launch_moments_small(const SmallBatch& b, int items, cudaStream_t s);
// alone: each problem has an SM to itself (they take one by their shared memory).
cudaError_t launch_basis_small(const SmallBatch& b, bool alone, cudaStream_t s);
cudaError_t launch_block_match_small(const SmallBatch& b, int items, size_t smem, cudaStream_t s);
cudaError_t launch_filter_small(const SmallBatch& b, int items, size_t smem, cudaStream_t s);
cudaError_t launch_reduce_small(const SmallBatch& b, int items, cudaStream_t s);

// ---- batched patch projection (project.cu): S = U^T * P * V per patch, 64 C coefficients in the
// order n = (i * 8 + j) * C + c; positions are linear top-left indices y * W + x (outside: NaN).
// Bytes of the split BF16 basis matrix (three pieces, both halves) that launch_project_split writes.
size_t project_pieces_bytes(int C);
cudaError_t launch_project_split(const double* d_b64, int C, void* d_pieces, cudaStream_t s);
// Tensor cores (C in {1, 3}); flag (may be null) gets bit 0 set if a wait for the tensor cores ran out.
cudaError_t launch_project_tc(const uint8_t* img, int H, int W, int C, const int32_t* pos, long long n,
                              const void* d_pieces, float* coef, int* flag, cudaStream_t s);
// Structured per-slice FP32 form on the CUDA cores.
cudaError_t launch_project_simt(const uint8_t* img, int H, int W, int C, const int32_t* pos, long long n,
                                const double* d_b64, float* coef, cudaStream_t s);

// ---- MRI volumes (volume.cu): Alg. 1 on 4 x 4 x 4 cubes of a D x H x W uint8 volume, the t-SVD
// tube along z (cube P[i][j][k] = v[z + k][y + i][x + j]); linear indices (z H + y) W + x.
struct VolGeo {
    int D, H, W;
    int s, win, K;
    int nrz, nry, nrx;       // references per axis
    int npz, npy, npx;       // candidate positions per axis
    int wnz, wny, wnx;       // window extent per axis
};
VolGeo make_vol_geo(int D, int H, int W, int s, int win, int K);
int volume_max_window();
cudaError_t launch_block_match_volume(const uint8_t* vol, const VolGeo& g, int32_t* idx, cudaStream_t s);
// uint64 [2][4][4][4][4]: rows R[a][a'][c][c'] then columns Q[b][b'][c][c'] of the reference cubes.
cudaError_t launch_volume_moments(const uint8_t* vol, const VolGeo& g, unsigned long long* d_mom, cudaStream_t s);
// HOST: canonical bases from the moments: b64 [2 (U, V)][4 slices][4][4] complex (re, im), slice 3 the
// conjugate of slice 1; returns the smallest relative eigen-gap over the slices 0..2 of U and V.
double volume_bases_host(const unsigned long long* mom, double* b64);
// Full second moment M (64 x 64) and sums S (64) of the reference cubes (uint64, exact), for the noise
// estimate; entry order u = (a * 4 + b) * 4 + c.
cudaError_t launch_volume_full_moment(const uint8_t* vol, const VolGeo& g, unsigned long long* d_M,
                                      unsigned long long* d_S, cudaStream_t s);
struct VolFilterArgs {
    const uint8_t* vol;
    VolGeo g;
    const int32_t* idx;      // [N][K]
    const double* basis64;   // device copy of the host bases
    float tau32;
    double tau64;
    float band_rel, band_abs;
    const float* w_in;       // optional per-group weights
    int agg_mode;
    float* num;              // D H W, zeroed by the caller
    float* den;
    uint32_t* mask_out;      // optional, 2 K words per group (bit m * 64 + (i * 4 + j) * 4 + k)
    float* weights_out;      // optional
    const int* dense;        // optional: volume_filter_kernel works only where it is set, volume_group_kernel where not
};
bool volume_filter_fits(const VolGeo& g);
cudaError_t launch_volume_filter(const VolFilterArgs& a, cudaStream_t s);
cudaError_t launch_volume_finalize(const float* num, const float* den, long long n, float* out, cudaStream_t s);

// Volume filter on projection planes (volume_group.cu): the projected cube at every position of the z planes
// pz0 .. pz0 + nz - 1 of positions (64 floats, coefficient order) and its squared norm, gathered by one
// warp per group; num and den as launch_volume_filter. mask_out words are cleared by the caller.
struct VolPlaneArgs {
    const uint8_t* vol;
    int D, H, W, pz0;
    const double* basis64;
    float* coef;             // [nz][H - 3][W - 3][64]
    float* pn;               // [nz][H - 3][W - 3]
    int* sample;             // optional: three words, zeroed before the first band; nothing is done where [2] is set
};
// With f, 128 sampled groups of it (K 16 or 32) set a.sample[2] if they keep more rows of coefficients than most in
// the mean.
cudaError_t launch_volume_plane(const VolPlaneArgs& a, int nz, const VolFilterArgs* f, int most, cudaStream_t s);
struct VolGroupArgs {
    VolFilterArgs f;
    const float* coef;
    const float* pn;
    int pz0;                 // first z plane of the planes
    int tz0;                 // first tile plane
    void* rec;               // volume_group_rec_bytes(g, tile planes)
};
bool volume_group_fits(const VolGeo& g);
// Mean rows of coefficients a group keeps up to which planes and group filter are the faster way (kEveryRow: at any).
int volume_rows_limit(const VolGeo& g);
int volume_tiles_z(const VolGeo& g);
int volume_tiles_plane(const VolGeo& g);
// Position planes [z0, z1) that the tile planes [t0, t1) gather from.
void volume_band(const VolGeo& g, int t0, int t1, int& z0, int& z1);
size_t volume_group_rec_bytes(const VolGeo& g, int tz);
cudaError_t launch_volume_group(const VolGroupArgs& a, int tz, cudaStream_t s);

// ---- hyperspectral cubes (cube.cu): Alg. 1 with C = N bands, one Haar slot of a group at a time
struct CubeArgs {
    const uint8_t* img;      // H x W x N uint8
    Geo g;                   // g.C = N
    const int32_t* idx;      // [groups][K]
    const float* basis32;    // basis32_floats(N) floats, cube layout
    const double* basis64;   // [2][N][8][8] complex
    float tau32;
    double tau64;
    float band_rel, band_abs; // guard band: |S| within band_rel ||G||_F + band_abs of tau -> FP64 decision
    const float* w_in;       // optional per-group weights
    int agg_mode;
    float* scratch;          // grid x K x 64 N floats (spatial Haar slots per CTA)
    float* num;              // H x W x N, zeroed by the launcher
    float* den;              // H x W, zeroed by the launcher
    float* out;              // H x W x N = num / den
    uint32_t* mask_out;      // optional: ceil(K 64 N / 32) words per group (bit (m 64 + p) N + c)
    float* weights_out;      // optional
    float* coef_out;         // optional: K 64 N floats per group
};
size_t cube_smem_bytes(int C, int K);
// CTAs of the persistent cube filter (a few per SM, at most one per group).
int cube_grid(int C, int K, int64_t ngroups);
cudaError_t launch_cube_filter(const CubeArgs& a, int grid, cudaStream_t s);

// ---- sigma adjustment (moments.cu)
// Rank position a = 1 + #{f : lambda_f < lambda_{K/2}} of each sampled group (Sec. III-D).
cudaError_t launch_group_rank(const uint8_t* img, const Geo& g, const int32_t* idx, int ngroups, int32_t* ranks,
                              cudaStream_t s);

}  // namespace htsvd
