// Block matching on the tensor cores (same grouping as bm_tile, bit for bit).
//
// The cross terms <v, r> of SSD = S_vv(v) - 2 <v, r> + S_vv(r) are a contraction of 128 reference
// patches (M) with the candidate patches of a row of positions (N), K = 64 pixels per plane. The planes
// are centred integers in FP16 (gray, G, R, B: x - 128; R+G+B: x - 383), so every product is exact, and
// |sum| <= 64 * 383^2 < 2^24 keeps the FP32 sums exact integers. Under green-channel matching both
// planes are contracted at once (K = 128): a reference's row holds its own plane and zeros for the other.
//
// B needs no im2col of patches: shared memory holds for every pixel the 16-byte strip of the 8 pixels
// starting there, so a candidate's K chunk i is the strip one image row further down, eight
// neighbouring candidates are one 128-byte core matrix, and all rows of candidates read the same strips.
//
// One CTA (two per SM) takes 128 references: 4 x 32 of them, or 8 x 16 where the rows of candidates of
// the former are too long; warps 0 .. 3 = TMEM lane quarters, each a 4 x 8 block, thread = reference; a
// fifth warp issues the MMAs, a row of candidates ahead. Each thread reads its reference's row of the
// accumulator, adds S_vv, and appends the candidates below its threshold to its buffer in shared memory
// as 32-bit keys (SSD << ib | window index). When a buffer holds 32 keys, every lane of the warp sorts its
// own 32 in registers (a compare-exchange network: 32 references per instruction) and merges them into
// its sorted list of the 32 smallest, whose K-th key is the new threshold.
// Keys hold SSD < 2^(32 - ib); a reference with fewer than K - 1 candidates below that (planes that
// differ by a hundred grey levels everywhere) is matched again over 64-bit keys by its warp.
//
// What bounds it: the selection, about 1,400 warp instructions per reference (the CUDA-core kernel takes
// 11,000); the MMAs are 0.4 ms of the 4.5 ms of a 3840 x 2160 RGB frame (stride 3, window 31, K 32), which
// took 11.0 ms on the CUDA cores. 512^2 RGB (stride 2): 0.64 -> 0.23 ms; 1080p gray: 1.53 -> 0.70 ms; per
// 1080p frame of a clip over three frames: 6.3 -> 2.0 ms. (Cutting a full buffer back by a bisection per
// lane instead of the sort took 17.3 ms per 3840 x 2160 frame: 2,500 instructions per reference.) The rule
// that picks it, with both sides measured: bm_tc_scratch.

constexpr int BT_REFS = 128;                    // references per tile (MMA rows)
constexpr int BT_THREADS = BT_REFS + 32;        // a thread per reference, and the issuing warp
constexpr int BT_SR = 16;                       // strip rows held at most (9 rows of candidates)
constexpr int BT_CAP = 48;                      // keys buffered per reference (32 + a step of 16 candidates)
constexpr int BT_KEY = 33 * 4;                  // bytes between a reference's buffered keys
constexpr int BT_ACC = 128;                     // TMEM columns per accumulator (two accumulators)

__host__ __device__ inline int bt_planes(int mode, int C) {
    if (C == 1) return 1;
    return mode == MM_FULL ? C : (mode == MM_GCP ? 2 : 1);
}

struct BtLayout {
    int a, strips, svv, buf, bar, total;
};
__host__ __device__ inline BtLayout bt_layout(int npl, int nsv, int XP, int SR) {
    BtLayout L;
    int o = 0;
    L.a = o; o += npl * 8 * BT_REFS * 16;
    L.strips = o; o += npl * SR * XP * 16;
    L.svv = o; o += nsv * (SR - PS + 1) * XP * 4;
    L.buf = o; o += 4 * BT_CAP * 33 * 4;
    L.bar = (o + 15) & ~15; o = L.bar + 48;
    L.total = o;
    return L;
}

// Centred planes (FP16) and box sums of their squares (FP32, exact) of one frame. Plane order: gray | G |
// G, R+G+B | R, G, B. Box sums: one per plane under green-channel matching, else one over all planes.
struct BtPrep {
    const uint8_t* img;
    int H, W, C, mode;
    __half* planes;          // [npl][H][pitch]
    float* svv;              // [nsv][H - 7][pitch]
    int pitch;
};

constexpr int BP_X = 64, BP_Y = 16;

template <int NPL, bool GCP>
__global__ void __launch_bounds__(256) bt_prep_kernel(BtPrep a) {
    __shared__ short v[NPL][BP_Y + PS - 1][BP_X + PS];
    __shared__ int hs[GCP ? 2 : 1][BP_Y + PS - 1][BP_X];
    const int x0 = blockIdx.x * BP_X, y0 = blockIdx.y * BP_Y, tid = threadIdx.x;
    constexpr int ROWS = BP_Y + PS - 1, COLS = BP_X + PS - 1;
    for (int t = tid; t < ROWS * COLS; t += 256) {
        const int r = t / COLS, c = t - r * COLS;
        const int y = y0 + r, x = x0 + c;
        short p[NPL];
#pragma unroll
        for (int k = 0; k < NPL; ++k) p[k] = 0;
        if (y < a.H && x < a.W) {
            const uint8_t* px = a.img + ((size_t)y * a.W + x) * a.C;
            if constexpr (GCP) {
                p[0] = (short)px[1] - 128;
                p[1] = (short)((int)px[0] + (int)px[1] + (int)px[2] - 383);
            } else if constexpr (NPL == 3) {
                p[0] = (short)px[0] - 128;
                p[1] = (short)px[1] - 128;
                p[2] = (short)px[2] - 128;
            } else {
                p[0] = (short)px[a.C == 1 ? 0 : 1] - 128;
            }
            if (r < BP_Y && c < BP_X) {
#pragma unroll
                for (int k = 0; k < NPL; ++k)
                    a.planes[((size_t)k * a.H + y) * a.pitch + x] = __short2half_rn(p[k]);
            }
        }
#pragma unroll
        for (int k = 0; k < NPL; ++k) v[k][r][c] = p[k];
    }
    __syncthreads();
    for (int t = tid; t < ROWS * BP_X; t += 256) {
        const int r = t / BP_X, c = t - r * BP_X;
        int s[GCP ? 2 : 1] = {};
#pragma unroll
        for (int k = 0; k < NPL; ++k)
#pragma unroll
            for (int j = 0; j < PS; ++j) s[GCP ? k : 0] += (int)v[k][r][c + j] * (int)v[k][r][c + j];
#pragma unroll
        for (int k = 0; k < (GCP ? 2 : 1); ++k) hs[k][r][c] = s[k];
    }
    __syncthreads();
    for (int t = tid; t < BP_Y * BP_X; t += 256) {
        const int r = t / BP_X, c = t - r * BP_X;
        if (y0 + r > a.H - PS || x0 + c > a.W - PS) continue;
#pragma unroll
        for (int k = 0; k < (GCP ? 2 : 1); ++k) {
            int s = 0;
#pragma unroll
            for (int i = 0; i < PS; ++i) s += hs[k][r + i][c];
            a.svv[((size_t)k * (a.H - PS + 1) + y0 + r) * a.pitch + x0 + c] = (float)s;
        }
    }
}

struct BtArgs {
    BMArgs b;
    const __half* planes;    // frame f0's planes; frames framestride_p apart
    const float* svv;
    long long fstride_p, fstride_s;
    int pitch;
    int XP;                  // padded candidates per row (multiple of 16)
    int SR;                  // strip rows held
    int TX;                  // references per tile row (32 or 16)
    int ib;                  // index bits of a key
    int* timeout;            // set (host memory) if a wait for the tensor cores runs out
    int give_up;             // every wait counts as run out (tests)
};

__device__ __forceinline__ void bt_tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Appends key at shared address ptr (which moves on) if the candidate is valid and d <= t. Predicated.
__device__ __forceinline__ void bt_append(uint32_t& ptr, uint32_t key, float d, float t, uint32_t mask, uint32_t bit) {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b32 m;\n\tand.b32 m, %4, %5;\n\tsetp.ne.b32 q, m, 0;\n\t"
        "setp.le.and.f32 p, %2, %3, q;\n\t@p st.shared.u32 [%0], %1;\n\t@p add.u32 %0, %0, 132;\n\t}"
        : "+r"(ptr)
        : "r"(key), "f"(d), "f"(t), "r"(mask), "r"(bit)
        : "memory");
}

// Merges the first 32 keys buffered at col .. ptr into the lane's sorted list and moves the rest down; the
// threshold drops to the K-th smallest key's.
__device__ __forceinline__ void bt_flush(uint32_t (&list)[32], uint32_t& ptr, float& thr, uint32_t col, int K, int ib,
                                         float srr) {
    uint32_t b[32];
    const uint32_t used = ptr - col;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        uint32_t k;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(k) : "r"(col + BT_KEY * i) : "memory");
        b[i] = BT_KEY * i < used ? k : ~0u;
    }
#pragma unroll
    for (int i = 0; i < BT_CAP - 32; ++i) {
        uint32_t k;
        asm volatile("ld.shared.u32 %0, [%1];" : "=r"(k) : "r"(col + BT_KEY * (32 + i)) : "memory");
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(col + BT_KEY * i), "r"(k) : "memory");
    }
    ptr = col + (used > 32u * BT_KEY ? used - 32u * BT_KEY : 0u);
    bt_sort(b);
    bt_merge(list, b);
    const uint32_t kth = K == 32 ? list[31] : K == 16 ? list[15] : K == 8 ? list[7] : K == 4 ? list[3] : list[1];
    // K keys have an SSD of at most kth's; a later candidate with that SSD has a larger index
    if (kth != ~0u) thr = (float)(kth >> ib) - 1.f - srr;
}

// The reference's K - 1 smallest (SSD, linear index) keys over all candidates, by the whole warp with
// 64-bit keys (lane l < K - 1 returns the l-th). Only for references whose keys outgrow 32 bits.
template <int NPL, bool GCP>
__device__ __noinline__ unsigned bt_wide(const BtArgs& A, int ry, int rx, bool green, unsigned long long* buf,
                                         int lane) {
    const BMArgs& a = A.b;
    const Geo& g = a.g;
    const int nfr = a.nfr > 0 ? a.nfr : 1, fsref = a.nfr > 0 ? a.fref - a.f0 : 0;
    const int wy0 = win_start(ry, g.npy, g.win), wx0 = win_start(rx, g.npx, g.win);
    const int p0 = GCP ? (green ? 0 : 1) : 0, p1 = GCP ? p0 + 1 : NPL;
    Select S;
    S.list = ~0ull;
    S.thr = ~0ull;
    S.buf = buf;
    S.cnt = 0;
    const int nw = g.wny * g.wnx;
    for (int fs = 0; fs < nfr; ++fs)
        for (int c0 = 0; c0 < nw; c0 += 32) {
            const int c = c0 + lane;
            unsigned long long key = ~0ull;
            if (c < nw) {
                const int py = wy0 + c / g.wnx, px = wx0 + c % g.wnx;
                if (fs != fsref || py != ry || px != rx) {
                    int ssd = 0;
                    for (int p = p0; p < p1; ++p)
                        for (int i = 0; i < PS; ++i) {
                            const __half* cv = A.planes + fs * A.fstride_p + ((size_t)p * g.H + py + i) * A.pitch + px;
                            const __half* rv = A.planes + fsref * A.fstride_p + ((size_t)p * g.H + ry + i) * A.pitch + rx;
#pragma unroll
                            for (int j = 0; j < PS; ++j) {
                                const int d = __half2int_rn(cv[j]) - __half2int_rn(rv[j]);
                                ssd += d * d;
                            }
                        }
                    const unsigned koff = a.nfr > 0 ? (unsigned)(a.f0 + fs) * (unsigned)(g.H * g.W) : 0u;
                    key = make_key(ssd, py, px, g.W, koff);
                }
            }
            sel_offer(S, key, g.K, lane);
        }
    if (S.cnt > 0) sel_merge(S, g.K, lane);
    __syncwarp();
    return (unsigned)(S.list & 0xffffffffull);
}

template <int NPL, bool GCP>
__global__ void __launch_bounds__(BT_THREADS, 2) block_match_tc_kernel(const __grid_constant__ BtArgs A) {
    extern __shared__ __align__(1024) unsigned char sm[];
    constexpr int NSV = GCP ? 2 : 1;
    const BMArgs& a = A.b;
    const Geo& g = a.g;
    const BtLayout L = bt_layout(NPL, NSV, A.XP, A.SR);
    const int tid = threadIdx.x, warp = __shfl_sync(FULL, tid >> 5, 0), lane = tid & 31;
    uint4* sA = reinterpret_cast<uint4*>(sm + L.a);
    uint4* strips = reinterpret_cast<uint4*>(sm + L.strips);
    float* svs = reinterpret_cast<float*>(sm + L.svv);
    uint32_t* buf = reinterpret_cast<uint32_t*>(sm + L.buf) + (warp & 3) * BT_CAP * 33;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + L.bar);            // full[2], empty[2]
    uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + L.bar + 32);
    volatile int* abort_word = reinterpret_cast<volatile int*>(sm + L.bar + 36);
    const int nfr = a.nfr > 0 ? a.nfr : 1, fsref = a.nfr > 0 ? a.fref - a.f0 : 0;

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&bars[i]), 1);
            mbar_init(smem_u32(&bars[2 + i]), 4);
        }
        *abort_word = A.give_up;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(2 * BT_ACC)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }

    // this thread's reference (the last one again where the tile leaves the grid)
    const int TX = A.TX, TY = BT_REFS / TX, bx = TX / 8;
    const int iy0 = blockIdx.y * TY, ix0 = blockIdx.x * TX;
    const int wb = warp & 3;                                        // 4 x 8 block of references
    const int iyr = iy0 + 4 * (wb / bx) + (lane >> 3), ixr = ix0 + 8 * (wb % bx) + (lane & 7);
    const bool mine = iyr < g.nry && ixr < g.nrx;
    const int iy = min(iyr, g.nry - 1), ix = min(ixr, g.nrx - 1);
    const int ry = ref_pos(iy, g.s, g.H), rx = ref_pos(ix, g.s, g.W);
    const int wy0 = win_start(ry, g.npy, g.win), wx0 = win_start(rx, g.npx, g.win);
    // candidate rows and columns of the tile
    const int Y0 = win_start(ref_pos(iy0, g.s, g.H), g.npy, g.win);
    const int Y1 = win_start(ref_pos(min(iy0 + TY, g.nry) - 1, g.s, g.H), g.npy, g.win) + g.wny;
    const int X0 = win_start(ref_pos(ix0, g.s, g.W), g.npx, g.win);
    const int X1 = win_start(ref_pos(min(ix0 + TX, g.nrx) - 1, g.s, g.W), g.npx, g.win) + g.wnx;
    const int XN = (X1 - X0 + 15) & ~15;                            // candidates per MMA row

    // plane choice (Eq. GCP distance on the reference patch) and the A row
    bool green = true;
    if (tid < BT_REFS) {
        if constexpr (GCP) {
            int r2 = 0, g2 = 0, b2 = 0;
            for (int i = 0; i < PS; ++i) {
                const uint8_t* px = a.img + ((size_t)(ry + i) * g.W + rx) * 3;
#pragma unroll
                for (int j = 0; j < PS; ++j) {
                    const int rr = px[3 * j], gg = px[3 * j + 1], bb = px[3 * j + 2];
                    r2 += rr * rr;
                    g2 += gg * gg;
                    b2 += bb * bb;
                }
            }
            const double lhs = a.gamma2 * (double)g2;
            green = (lhs >= (double)r2) && (lhs >= (double)b2);
        }
        for (int p = 0; p < NPL; ++p)
            for (int i = 0; i < PS; ++i) {
                uint32_t w[4] = {0u, 0u, 0u, 0u};
                if (!GCP || (p == 0) == green) {
                    const unsigned short* src = reinterpret_cast<const unsigned short*>(
                        A.planes + fsref * A.fstride_p + ((size_t)p * g.H + ry + i) * A.pitch + rx);
#pragma unroll
                    for (int j = 0; j < 4; ++j) w[j] = (uint32_t)src[2 * j] | ((uint32_t)src[2 * j + 1] << 16);
                }
                sA[(p * PS + i) * BT_REFS + tid] = make_uint4(w[0], w[1], w[2], w[3]);
            }
    }
    const int svp = GCP ? (green ? 0 : 1) : 0;
    const int np_rows = g.H - PS + 1;
    const float srr = A.svv[fsref * A.fstride_s + ((size_t)svp * np_rows + ry) * A.pitch + rx];
    const int ib = A.ib;
    const uint32_t mul = 1u << ib;
    // largest SSD a key holds (and the exact range of the float-to-integer step below)
    const float lim = (float)min((1u << (32 - ib)) - 2u, (1u << 23) - 2u);
    float thr = lim - srr;                            // S_vv(v) - 2 <v, r> <= thr
    const uint32_t col = smem_u32(buf) + 4u * lane;   // this reference's buffered keys, BT_KEY bytes apart
    uint32_t ptr = col;
    uint32_t list[32];                                // its smallest keys so far, ascending
#pragma unroll
    for (int i = 0; i < 32; ++i) list[i] = ~0u;
    const int xlo = wx0 - X0, xhi = xlo + g.wnx;      // this reference's candidate columns
    int cbeg = xlo, cend = xhi;                       // the warp's
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        cbeg = min(cbeg, __shfl_xor_sync(FULL, cbeg, o));
        cend = max(cend, __shfl_xor_sync(FULL, cend, o));
    }
    cbeg &= ~3;                                       // box sums are read four at a time, in steps of 16 candidates
    cbeg = min(cbeg, A.XP - ((cend - cbeg + 15) & ~15));
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const uint32_t idesc = idesc_f16(128, XN);
    const uint32_t a_addr = smem_u32(sA), b_addr = smem_u32(strips);
    const uint32_t LBO_B = (uint32_t)A.XP * 16u;

    uint32_t it = 0;                                  // rows of candidates done (accumulator it & 1)
    uint32_t issued = 0;                              // the issuing lane: rows whose MMAs are committed
    bool ok = true;
    for (int fs = 0; fs < nfr && ok; ++fs) {
        const __half* fp = A.planes + fs * A.fstride_p;
        const float* fsv = A.svv + fs * A.fstride_s;
        for (int yb = Y0; yb < Y1 && ok; yb += A.SR - PS + 1) {
            const int rows = min(A.SR - PS + 1, Y1 - yb);
            // strips of image rows yb .. yb + rows + 6: a pair of neighbouring strips from five words
            const int pairs = XN / 2;
            for (int t = tid; t < NPL * (rows + PS - 1) * pairs; t += BT_THREADS) {
                const int pr = t / pairs, xp = t - pr * pairs;
                const int p = pr / (rows + PS - 1), r = pr - p * (rows + PS - 1);
                const int x = X0 + 2 * xp;
                const uint32_t* src = reinterpret_cast<const uint32_t*>(fp + ((size_t)p * g.H + yb + r) * A.pitch) + (x >> 1);
                // (words past the image feed only candidates that no reference looks at)
                uint32_t h[5], o[4];
#pragma unroll
                for (int e = 0; e < 5; ++e) h[e] = __ldg(src + e);
#pragma unroll
                for (int e = 0; e < 4; ++e) o[e] = __byte_perm(h[e], h[e + 1], 0x5432);
                uint4* d = strips + (p * A.SR + r) * A.XP + 2 * xp;
                const bool odd = x & 1;
                d[0] = odd ? make_uint4(o[0], o[1], o[2], o[3]) : make_uint4(h[0], h[1], h[2], h[3]);
                d[1] = odd ? make_uint4(h[1], h[2], h[3], h[4]) : make_uint4(o[0], o[1], o[2], o[3]);
            }
            for (int t = tid; t < NSV * rows * XN; t += BT_THREADS) {
                const int pr = t / XN, x = t - pr * XN;
                const int p = pr / rows, r = pr - p * rows;
                svs[(r * NSV + p) * A.XP + x] = fsv[((size_t)p * np_rows + yb + r) * A.pitch + X0 + x];
            }
            fence_async_smem();
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
            if (warp == 4) {
                // ---- the MMAs: row j of candidates into accumulator (it + j) & 1
                if (lane == 0) {
                    for (int j = 0; j < rows; ++j) {
                        const uint32_t n = it + j, acc = n & 1;
                        if (n >= 2 && !mbar_wait_or_abort(smem_u32(&bars[2 + acc]), ((n >> 1) & 1) ^ 1, abort_word)) break;
                        tc_fence_after();
                        uint32_t on = 0;
#pragma unroll
                        for (int s = 0; s < NPL * 4; ++s) {
                            const int p = s / 4, i = 2 * (s % 4);
                            const uint64_t ad = smem_desc(a_addr + (uint32_t)(p * PS + i) * (BT_REFS * 16), BT_REFS * 16, 128);
                            const uint64_t bd = smem_desc(b_addr + (uint32_t)((p * A.SR + j + i) * A.XP) * 16u, LBO_B, 128);
                            mma_f16(tmem + acc * BT_ACC, ad, bd, idesc, on);
                            on = 1;
                        }
                        mma_commit(smem_u32(&bars[acc]));
                        issued = n + 1;
                    }
                }
                __syncwarp();
            } else {
                // ---- the candidates of this warp's references
                for (int j = 0; j < rows; ++j) {
                    const uint32_t n = it + j, acc = n & 1;
                    const bool got = mbar_wait_or_abort(smem_u32(&bars[acc]), (n >> 1) & 1, abort_word);
                    if (__any_sync(FULL, !got)) break;
                    tc_fence_after();
                    const int wy = yb + j - wy0;
                    const bool in = wy >= 0 && wy < g.wny;
                    if (__any_sync(FULL, in)) {
                        const uint32_t kb = (uint32_t)((fs * g.wny + wy) * g.wnx - xlo);
                        const float* sv = svs + (j * NSV + svp) * A.XP;
                        const uint32_t ta = tmem + acc * BT_ACC + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
                        for (int c0 = cbeg; c0 < cend; c0 += 16) {
                            float v[16];
                            bt_tmem_ld16(ta + c0, v);
                            const int lo = min(max(xlo - c0, 0), 16), hi = min(max(xhi - c0, 0), 16);
                            const uint32_t mask = in ? (1u << hi) - (1u << lo) : 0u;
                            const uint32_t kc = kb + (uint32_t)c0;
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float4 q = *reinterpret_cast<const float4*>(sv + c0 + 4 * e);
                                const float s4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                                for (int u = 0; u < 4; ++u) {
                                    const float d = fmaf(-2.f, v[4 * e + u], s4[u]);
                                    // SSD + 2^23: the integer SSD in the mantissa bits
                                    const uint32_t key = __float_as_uint((d + srr) + 8388608.f) * mul + (kc + 4 * e + u);
                                    bt_append(ptr, key, d, thr, mask, 1u << (4 * e + u));
                                }
                            }
                            if (__any_sync(FULL, ptr > col + (BT_CAP - 16) * BT_KEY)) bt_flush(list, ptr, thr, col, g.K, ib, srr);
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&bars[2 + acc]));
                }
            }
            it += rows;
            __syncthreads();
            if (*abort_word) ok = false;
        }
    }
    if (!ok) {
        // A wait ran out: report it, and let the MMAs in flight finish (bounded) before the tensor memory is
        // released. The last commit covers all of them, and its barrier is at most that one phase behind: row
        // issued - 1 was issued after row issued - 3 of the same accumulator had been read. The groups below
        // hold what was found, or the reference alone.
        if (tid == 0) *A.timeout = 1;
        if (warp == 4 && lane == 0 && issued > 0)
            mbar_wait_bounded(smem_u32(&bars[(issued - 1) & 1]), ((issued - 1) >> 1) & 1);
    }
    if (warp < 4) {
        while (__any_sync(FULL, ptr != col)) bt_flush(list, ptr, thr, col, g.K, ib, srr);
        // ---- the groups: the list without the reference itself (SSD 0), as linear positions
        const uint32_t self = (uint32_t)((fsref * g.wny + (ry - wy0)) * g.wnx + rx - wx0);
        const uint32_t imask = mul - 1u;
        const int nw = g.wny * g.wnx;
        const int fo = a.nfr > 0 ? a.f0 * g.H * g.W : 0;
        bool past = false, enough = true;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 31; ++i) {
            past = past || list[i] == self;
            const uint32_t k = past ? list[i + 1] : list[i];
            if (i < g.K - 1) enough = enough && k != ~0u;
            const int w = (int)(k & imask);
            const int fs = w / nw, wr = w - fs * nw;
            const int dy = wr / g.wnx, dx = wr - dy * g.wnx;
            buf[i * 33 + lane] = (uint32_t)(fo + fs * g.H * g.W + (wy0 + dy) * g.W + wx0 + dx);
        }
        __syncwarp();
        const unsigned wide = __ballot_sync(FULL, mine && !enough), valid = __ballot_sync(FULL, mine);
        const int home = fo + fsref * g.H * g.W + ry * g.W + rx, gi = iy * g.nrx + ix;
        const unsigned none = ok ? 0u : wide;           // given up before the group was full: the reference alone
        for (int l = 0; l < 32; ++l) {
            if (!((valid >> l) & 1u)) continue;
            const int h = __shfl_sync(FULL, home, l), gl = __shfl_sync(FULL, gi, l);
            if (lane < g.K) a.idx[(size_t)gl * g.K + lane] = lane == 0 || ((none >> l) & 1u) ? h : (int32_t)buf[(lane - 1) * 33 + l];
        }
        __syncwarp();
        for (unsigned m = ok ? wide : 0u; m; m &= m - 1) {              // warp-uniform
            const int l = __ffs(m) - 1;
            const int qy = __shfl_sync(FULL, ry, l), qx = __shfl_sync(FULL, rx, l);
            const int gl = __shfl_sync(FULL, gi, l);
            const bool qg = __shfl_sync(FULL, (int)green, l) != 0;
            __syncwarp();
            const unsigned e = bt_wide<NPL, GCP>(A, qy, qx, qg, reinterpret_cast<unsigned long long*>(buf), lane);
            if (lane < g.K - 1) a.idx[(size_t)gl * g.K + 1 + lane] = (int32_t)e;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 4) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BT_ACC) : "memory");
    }
}
