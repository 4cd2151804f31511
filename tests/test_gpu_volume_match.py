"""Volume grouping with a thread per reference (window cubes of 4 to 6, 6,000 references or more) against the
FP64 oracle, index by index: windows, alignments, ties and the largest distances."""
import numpy as np
import pytest
import torch

import paper_2508_10307_gb300 as H
from oracle import htsvd_oracle as O
from paper_2508_10307_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,shape,window,K", [
    ("noise", (42, 46, 45), 4, 32),          # rows of every alignment
    ("noise", (43, 44, 48), 5, 32),
    ("noise", (45, 43, 46), 6, 16),
    ("noise", (42, 45, 47), 5, 2),           # not whole vectors of indices
    ("constant", (42, 43, 45), 6, 32),       # every distance ties: the lowest indices win
    ("binary", (42, 43, 45), 5, 8),          # the largest distances
])
def test_lane_grouping_matches_oracle(kind, shape, window, K):
    rng = np.random.default_rng(11)
    if kind == "constant":
        v = np.full(shape, 201, dtype=np.uint8)
    elif kind == "binary":
        v = (rng.integers(0, 2, shape) * 255).astype(np.uint8)
    else:
        v = synth.add_gaussian(synth.clean_volume(*shape, 4), 15.0, 4)
    prm = dict(ps=4, stride=2, window=window, K=K)
    _, info = H.denoise_volume(torch.from_numpy(v).cuda(), 10.0, prm, return_info=True)
    idx = info["idx"].cpu().numpy().astype(np.int64)
    n = idx.shape[0]
    assert n >= 6000
    pick = np.concatenate([np.arange(24), np.arange(n - 24, n), rng.choice(n, 250, replace=False)])
    assert np.array_equal(idx[pick], O.block_match_volume(v, prm, only=pick))
