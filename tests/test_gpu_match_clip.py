"""Tensor-core block matching of clips (groups from several frames) against the FP64 oracle's grouping, index by
index: first, middle and last frames, the key's index bits, and keys that outgrow 32 bits. Every frame here is large
enough for that path (at least 76 tiles of 128 references, at most 4,096 candidates over the frames)."""
import numpy as np
import pytest
import torch

import paper_2508_10307_gb300 as H
from oracle import htsvd_oracle as O
from paper_2508_10307_gb300 import synth

pytestmark = pytest.mark.gpu


def _check(clip, prm, T, rows=(0, 1, 40)):
    F, Hh, Ww, _ = clip.shape
    _, info = H.denoise_video(torch.from_numpy(clip).cuda(), 20.0, prm, T=T, return_info=True)
    idx = info["idx"].cpu().numpy().astype(np.int64)
    p = O.Params.of({k: ("gray" if v == "green" else v) for k, v in prm.items()})
    ys, xs = O.reference_positions(Hh, 8, p.stride), O.reference_positions(Ww, 8, p.stride)
    idx = idx.reshape(F, len(ys), len(xs), p.K)
    for t in sorted({0, F // 2, F - 1}):
        for r in sorted({*rows, len(ys) - 1}):
            ref = O._match_row_video(clip, t, int(ys[r]), xs, p, T)
            ref = ref[0] if isinstance(ref, tuple) else ref
            assert np.array_equal(idx[t, r], ref), f"frame {t}, reference row {r}"


@pytest.mark.parametrize("F,shape,T,stride,window,K,mode", [
    (3, (330, 340, 3), 1, 3, 31, 32, "auto"),        # 2,883 candidates: twelve index bits
    (5, (329, 333, 1), 2, 3, 28, 32, "auto"),        # 3,920 candidates
    (3, (331, 336, 3), 1, 3, 18, 8, "full"),
    (4, (330, 335, 3), 3, 3, 9, 16, "green"),
    (2, (260, 262, 3), 1, 2, 45, 4, "auto"),         # 4,050 candidates
])
def test_indices_match_oracle(F, shape, T, stride, window, K, mode):
    clean = synth.clean_image(shape[0], shape[1] + F, shape[2], 17)
    clip = np.stack([synth.add_gaussian(np.ascontiguousarray(clean[:, t:t + shape[1]]), 25.0, 17 + t) for t in range(F)])
    _check(clip, dict(stride=stride, window=window, K=K, match_mode=mode), T)


def test_distances_beyond_the_keys():
    rng = np.random.default_rng(5)
    clip = (rng.integers(0, 2, (3, 330, 330, 1)) * np.array([255, 120, 255])).astype(np.uint8)
    _check(np.ascontiguousarray(clip), dict(stride=3, window=31, K=32), 1, rows=(30, 60))
