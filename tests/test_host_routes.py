"""Rules that choose a kernel, looked at on the host."""
import pytest

import paper_2508_10307_gb300 as H


@pytest.mark.parametrize("D,H_,W,stride,window,K,want", [
    (176, 208, 176, 2, 5, 32, 1),
    (32, 32, 32, 2, 5, 32, 0),               # 3,375 references: too few
    (200, 200, 200, 3, 7, 32, 0),            # the footprint of a tile fills an SM's shared memory
    (850_000, 8, 8, 680, 5, 32, 0),          # 2,048 voxels an edge: 2^33, which is 0 in 32 bits
    (850_000, 8, 8, 680, 5, 2, 0),
    (1 << 24, 8, 8, 2048 * 3, 4, 8, 0),
])
def test_volume_planes_need_a_footprint_that_fits(D, H_, W, stride, window, K, want):
    assert H.load_library().htsvd_internal_volume_planes(D, H_, W, stride, window, K) == want
