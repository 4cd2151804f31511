"""Tensor-core block matching against the FP64 oracle's grouping, index by index, at the edges of its
tiles, keys and planes. Every image here is large enough for that path (at least 76 tiles of 128
references, 152 where the tiles are 8 x 16); reference rows are sampled to keep the oracle's share short."""
import numpy as np
import pytest
import torch

import paper_2508_10307_gb300 as H
from oracle import htsvd_oracle as O
from paper_2508_10307_gb300 import synth

pytestmark = pytest.mark.gpu


def _check(noisy, prm, rows):
    _, info = H.denoise(torch.from_numpy(noisy).cuda(), 20.0, prm, return_info=True)
    idx = info["idx"].cpu().numpy().astype(np.int64)
    p = O.Params.of({k: ("gray" if v == "green" else v) for k, v in prm.items()})
    ys = O.reference_positions(noisy.shape[0], 8, p.stride)
    xs = O.reference_positions(noisy.shape[1], 8, p.stride)
    idx = idx.reshape(len(ys), len(xs), p.K)
    for r in sorted({0, 1, len(ys) - 1, *rows}):
        ref, _, _ = O._match_row(noisy, int(ys[r]), xs, p)
        assert np.array_equal(idx[r], ref), f"reference row {r}"


@pytest.mark.parametrize("H_,W_,C,stride,window,K,mode", [
    (330, 331, 3, 3, 31, 32, "auto"),        # both planes, ragged tiles
    (257, 300, 3, 2, 32, 32, "auto"),        # 1,024 candidates: ten index bits
    (300, 420, 3, 3, 33, 16, "auto"),        # eleven index bits
    (330, 340, 3, 3, 18, 8, "full"),         # three planes
    (330, 340, 3, 3, 21, 4, "green"),
    (330, 333, 1, 3, 7, 2, "auto"),          # smallest windows: a row of candidates is shorter than a step
    (500, 660, 1, 4, 31, 32, "auto"),        # 8 x 16 references per tile
    (680, 700, 3, 5, 40, 32, "auto"),        # 8 x 16, rows of 128 candidates
])
def test_indices_match_oracle(H_, W_, C, stride, window, K, mode):
    noisy = synth.add_gaussian(synth.clean_image(H_, W_, C, 71), 25.0, 71)
    _check(noisy, dict(stride=stride, window=window, K=K, match_mode=mode), rows=(5, 17))


@pytest.mark.parametrize("kind", ["constant", "tiles", "binary", "saturated"])
def test_ties_and_extreme_values(kind):
    rng = np.random.default_rng(5)
    n = 330
    if kind == "constant":                   # every distance ties: the lowest indices win
        noisy = np.full((n, n, 3), 97, dtype=np.uint8)
    elif kind == "tiles":                    # a repeated 4 x 4 texture: ties at every multiple
        noisy = np.tile(rng.integers(0, 256, (4, 4, 3), dtype=np.uint8), (83, 83, 1))[:n, :n]
    elif kind == "binary":                   # distances beyond the 32-bit keys: the 64-bit pass
        noisy = (rng.integers(0, 2, (n, n, 1)) * np.array([255, 120, 255])).astype(np.uint8)
    else:                                    # extreme areas on the R+G+B plane: the largest products and box sums
        noisy = np.zeros((n, n, 3), dtype=np.uint8)
        noisy[:, n // 2:] = (255, 211, 255)
        noisy[::37, ::5] = rng.integers(0, 256, noisy[::37, ::5].shape, dtype=np.uint8)
    _check(np.ascontiguousarray(noisy), dict(stride=3, window=31, K=32), rows=(30, 60))


def test_image_of_a_million_rows():
    """More rows than a grid of the tensor-core form reaches: the other form groups it, as it did before."""
    h, w = 1_050_000, 16
    rng = np.random.default_rng(11)
    noisy = (np.arange(h)[:, None, None] // 64 % 200 + rng.integers(0, 40, (h, w, 1))).astype(np.uint8)
    _check(noisy, dict(stride=16, window=9, K=8), rows=(40_000, 65_000))
