"""Volume filter on projection planes (5,000 references or more) against the FP64 oracle at the edges of its
tiles, windows, slot counts and row lists. Bars as for the other volume tests: indices exact, masks exact (but
for coefficients the oracle finds within 1e-9 of tau), voxels within 1e-3."""
import numpy as np
import pytest
import torch

import paper_2508_10307_gb300 as H
from oracle import htsvd_oracle as O
from paper_2508_10307_gb300 import synth
from tests._common import PIX_TOL, max_abs, pack_masks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,prm,sigma", [
    ((39, 40, 38), dict(stride=2, window=5, K=32), 11.5),
    ((32, 34, 70), dict(stride=2, window=4, K=16, agg_mode="sparsity"), 9.0),   # two blocks of positions a row
    ((38, 39, 40), dict(stride=2, window=6, K=8), 20.0),
    ((40, 38, 39), dict(stride=2, window=3, K=4, tau_mult=2.0), 15.0),
    ((39, 38, 40), dict(stride=2, window=4, K=2), 11.5),
    ((38, 40, 39), dict(stride=2, window=5, K=32, tau_mult=0.3), 6.0),           # nearly every row kept
    ((56, 57, 58), dict(stride=3, window=7, K=32, tau_mult=40.0), 11.5),         # hardly a coefficient kept
])
def test_volume_filter_matches_oracle(shape, prm, sigma):
    _check(synth.add_gaussian(synth.clean_volume(*shape, 6), sigma, 6), dict(ps=4, **prm), sigma)


def _check(v, prm, sigma):
    r = O.denoise_volume(v, sigma, prm, keep_masks=True)
    out, info = H.denoise_volume(torch.from_numpy(v).cuda(), sigma, prm, return_info=True, masks=True, weights=True)
    assert len(r.idx) >= 5000
    assert np.array_equal(info["idx"].cpu().numpy().astype(np.int64), r.idx)
    om = pack_masks(r.masks)
    gm = info["masks"].cpu().numpy().view(np.uint32)[:, :om.shape[1]]
    amb = {(int(g), int(i)) for g, i in r.ambiguous}
    for g, wd in zip(*np.nonzero(om != gm)):
        d = int(om[g, wd]) ^ int(gm[g, wd])
        assert all((int(g), int(wd) * 32 + b) in amb for b in range(32) if (d >> b) & 1)
    np.testing.assert_allclose(info["weights"].cpu().numpy(), r.weights, rtol=1e-6)
    assert max_abs(out.cpu().numpy(), r.out) <= PIX_TOL


@pytest.mark.parametrize("K,agg,half", [(32, "uniform", 20), (16, "sparsity", 8), (16, "uniform", 39)])
def test_dense_volumes(K, agg, half):
    """Noise above the threshold in a part: the groups sampled decide which kernel filters the volume."""
    v = synth.add_gaussian(synth.clean_volume(44, 39, 38, 6), 4.0, 6)
    rng = np.random.default_rng(3)
    v[:, half:] = rng.integers(0, 256, v[:, half:].shape)
    _check(np.ascontiguousarray(v), dict(ps=4, stride=2, window=4, K=K, agg_mode=agg), 15.0)
