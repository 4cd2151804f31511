// Sorting 32 keys per lane in registers: a network of compare-exchanges that every lane runs on its own keys,
// so that a warp sorts 32 lists per instruction.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace htsvd {

__device__ __forceinline__ void bt_order(uint32_t& a, uint32_t& b) {
    const uint32_t lo = min(a, b), hi = max(a, b);
    a = lo;
    b = hi;
}
// Sorts 32 keys of the lane ascending (Batcher's odd-even merge sort, 191 compare-exchanges). Templates, so
// that every index is a constant and the keys stay in registers.
template <int P, int K>
__device__ __forceinline__ void bt_sort_step(uint32_t (&v)[32]) {
#pragma unroll
    for (int i = 0; i < 32 - K; ++i)
        if (i >= K % P && (i - K % P) % (2 * K) < K && i / (2 * P) == (i + K) / (2 * P)) bt_order(v[i], v[i + K]);
    if constexpr (K > 1) bt_sort_step<P, K / 2>(v);
}
template <int P>
__device__ __forceinline__ void bt_sort_from(uint32_t (&v)[32]) {
    bt_sort_step<P, P>(v);
    if constexpr (P < 16) bt_sort_from<2 * P>(v);
}
__device__ __forceinline__ void bt_sort(uint32_t (&v)[32]) { bt_sort_from<1>(v); }
// The 32 smallest of two sorted lists, sorted, into a.
__device__ __forceinline__ void bt_merge(uint32_t (&a)[32], const uint32_t (&b)[32]) {
#pragma unroll
    for (int i = 0; i < 32; ++i) a[i] = min(a[i], b[31 - i]);
#pragma unroll
    for (int k = 16; k >= 1; k >>= 1)
#pragma unroll
        for (int i = 0; i < 32; ++i)
            if ((i & k) == 0) bt_order(a[i], a[i + k]);
}

}  // namespace htsvd
