// Small images of a batch, one launch a phase: a block takes a work item (chunk of references, tile, pixel block) of
// one of the images, found by its place in the images' running totals. The images' description travels as a
// kernel parameter: nothing is copied to the device, and a captured launch holds it by value.
#pragma once
#include "kernels.h"

namespace htsvd {

// The image whose items (running totals P) include item w.
template <int SmallImage::*P>
__device__ __forceinline__ int small_find(const SmallBatch& B, int w) {
    int lo = 0, hi = B.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (B.im[mid].*P <= w) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}
__device__ __forceinline__ Geo small_geo(const SmallBatch& B, const SmallImage& m) {
    return make_geo(m.H, m.W, B.C, B.s, B.win, B.K);
}

}  // namespace htsvd
