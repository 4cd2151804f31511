"""Coefficients exported by the group filter on projection planes against the FP64 oracle's, within the band inside
which a threshold is decided again in FP64 (2^-19 of the group's norm)."""
import numpy as np
import pytest
import torch

import paper_2508_10307_gb300 as H
from oracle import htsvd_oracle as O
from paper_2508_10307_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,prm,sigma", [
    ((117, 122, 3), dict(stride=2, window=13, K=32), 25.0),
    ((125, 119, 3), dict(stride=2, window=12, K=16), 25.0),
    ((118, 131, 1), dict(stride=2, window=10, K=8), 25.0),
    ((117, 127, 3), dict(stride=2, window=9, K=2), 20.0),
    ((119, 121, 1), dict(stride=2, window=12, K=32), 30.0),
    ((117, 122, 3), dict(stride=2, window=13, K=32, tau_mult=1.5), 8.0),       # the tile kernel's, beside it
])
def test_coefficients_match_oracle(shape, prm, sigma):
    noisy = synth.add_gaussian(synth.clean_image(*shape, 53), sigma, 53)
    r = O.denoise(noisy, sigma, prm, keep_masks=True)
    _, info = H.denoise(torch.from_numpy(noisy).cuda(), sigma, prm, return_info=True, coeffs=True)
    assert len(r.idx) >= 3000 and np.array_equal(info["idx"].cpu().numpy(), r.idx)
    got = info["coeffs"].cpu().numpy().astype(np.float64)
    for lo in range(0, len(r.idx), 512):
        i = r.idx[lo:lo + 512]
        G = O.gather_groups(noisy.astype(np.float64), i, 8)
        S = O.forward_transform(G, r.U, r.V, O.haar_matrix(prm["K"]))
        lim = 2.0 ** -19 * np.sqrt((G ** 2).reshape(len(i), -1).sum(1))
        assert (np.abs(got[lo:lo + 512] - S).reshape(len(i), -1).max(1) <= lim).all()
