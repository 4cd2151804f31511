"""Group filter on projection planes against the FP64 oracle, at the edges of its tiles, its slot counts
and its row lists. Every image has at least 3,000 references, from which on the planes are used. The bars
are those of the parity tests: indices and masks exact (masks but for coefficients the oracle finds within
1e-9 of tau), pixels within 1e-3, gradients within 1e-4 of the largest."""
import numpy as np
import pytest
import torch

import paper_2508_10307_gb300 as H
from oracle import htsvd_oracle as O
from paper_2508_10307_gb300 import synth
from tests._common import PIX_TOL, max_abs, pack_masks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,prm,sigma", [
    ((117, 127, 3), dict(stride=2, window=9, K=2), 20.0),                      # ragged tiles, fewest slots
    ((116, 125, 3), dict(stride=2, window=11, K=4, agg_mode="sparsity"), 15.0),
    ((118, 131, 1), dict(stride=2, window=10, K=8), 25.0),
    ((125, 119, 3), dict(stride=2, window=12, K=16), 25.0),
    ((119, 121, 1), dict(stride=2, window=12, K=32, agg_mode="sparsity"), 30.0),
    ((117, 122, 3), dict(stride=2, window=13, K=32), 25.0),
    ((117, 122, 3), dict(stride=2, window=13, K=32, tau_mult=1.5), 8.0),       # long row lists, tiles left over
    ((117, 122, 1), dict(stride=2, window=13, K=16, tau_mult=1.0), 8.0),
    ((117, 122, 3), dict(stride=2, window=13, K=32, tau_mult=30.0), 25.0),     # hardly a coefficient kept
    ((121, 120, 3), dict(stride=2, window=9, K=8, tile=1), 20.0),              # tiles of one group
    ((121, 120, 3), dict(stride=2, window=9, K=16, tile=7), 20.0),
])
def test_group_filter_matches_oracle(shape, prm, sigma):
    clean = synth.clean_image(*shape, 53)
    noisy = synth.add_gaussian(clean, sigma, 53)
    r = O.denoise(noisy, sigma, {k: v for k, v in prm.items() if k != "tile"}, keep_masks=True)
    assert len(r.idx) >= 3000
    out, info = H.denoise(torch.from_numpy(noisy).cuda(), sigma, prm, return_info=True, masks=True, weights=True)
    assert np.array_equal(info["idx"].cpu().numpy(), r.idx)
    om = pack_masks(r.masks)
    gm = info["masks"].cpu().numpy().view(np.uint32)[:, :om.shape[1]]
    amb = {(int(g), int(i)) for g, i in r.ambiguous}
    for g, wd in zip(*np.nonzero(om != gm)):
        d = int(om[g, wd]) ^ int(gm[g, wd])
        assert all((int(g), int(wd) * 32 + b) in amb for b in range(32) if (d >> b) & 1)
    np.testing.assert_allclose(info["weights"].cpu().numpy(), r.weights, rtol=1e-6)
    assert max_abs(out.cpu().numpy(), r.out) <= PIX_TOL


@pytest.mark.parametrize("C,K,mult", [(3, 32, 0.0), (1, 16, 0.0), (3, 8, 1.5), (3, 32, 1.2), (1, 32, 1.0)])
def test_group_filter_gradients_match_oracle(C, K, mult):
    x = synth.add_gaussian_float(synth.clean_image(118, 121, C, 7), 20.0, 7)
    prm = dict(stride=2, window=9, K=K, tau_mult=mult)
    rng = np.random.default_rng(4)
    r = O.denoise(x.astype(np.float64), 20.0, prm, keep_masks=True)
    w = rng.uniform(0.5, 1.5, size=len(r.idx))
    gout = rng.standard_normal(x.shape)
    gx_o, gw_o = O.denoise_fixed_vjp(x.astype(np.float64), gout, r.idx, r.masks, r.U, r.V, w, 8)
    xt, wt = torch.from_numpy(x).cuda(), torch.from_numpy(w.astype(np.float32)).cuda()
    out, info = H.denoise_f32(xt, 20.0, prm, w=wt, return_info=True)
    gx, gw = H.denoise_vjp(xt, 20.0, info["idx"], wt, out, torch.from_numpy(gout.astype(np.float32)).cuda(), prm)
    assert np.abs(gx.cpu().numpy() - gx_o).max() <= 1e-4 * np.abs(gx_o).max()
    assert np.abs(gw.cpu().numpy() - gw_o).max() <= 1e-4 * max(1.0, np.abs(gw_o).max())


@pytest.mark.parametrize("C,sigma,mult", [(3, 20.0, 0.0), (1, 10.0, 1.2)])
def test_group_filter_of_a_clip_matches_oracle(C, sigma, mult):
    clean = synth.clean_image(118, 124, C, 9)
    vid = np.stack([synth.add_gaussian(np.roll(clean, t, axis=1), sigma, 9 + t) for t in range(2)])
    prm = dict(stride=2, window=7, K=16, tau_mult=mult)
    out = H.denoise_video(torch.from_numpy(vid).cuda(), sigma, prm, T=1)
    ref, _ = O.denoise_video(vid, sigma, prm, T=1)
    assert max_abs(out.cpu().numpy(), ref) <= PIX_TOL


@pytest.mark.parametrize("n", [1, 20])
def test_batch_of_uneven_images_equals_single_calls(n):
    """More images than lanes, small ones among those that use the planes. A batch may cut its images into
    other filter tiles than a single call does: FP32 sums in another order."""
    prm = dict(stride=2, window=7, K=8)
    sizes = ([(40, 300), (125, 130), (33, 9 + 8), (117, 122), (64, 64)] * 4)[:n]
    xs = [torch.from_numpy(synth.add_gaussian(synth.clean_image(h, w, 3, 5 + i), 20.0, i)).cuda()
          for i, (h, w) in enumerate(sizes)]
    sig = [10.0 + 2 * i for i in range(n)]
    for x, s, o in zip(xs, sig, H.denoise_batch(xs, sig, prm)):
        assert max_abs(o.cpu().numpy(), H.denoise(x, s, prm).cpu().numpy()) <= PIX_TOL


@pytest.mark.parametrize("tile", [-1, 17, 20])
def test_batch_takes_any_tile_edge(tile):
    x = torch.from_numpy(synth.add_gaussian(synth.clean_image(117, 122, 1, 5), 20.0, 5)).cuda()
    prm = dict(stride=1, window=5, K=8)
    out, = H.denoise_batch([x], [20.0], dict(prm, tile=tile))
    assert max_abs(out.cpu().numpy(), H.denoise(x, 20.0, prm).cpu().numpy()) <= PIX_TOL


@pytest.mark.parametrize("shape,K,mult", [
    ((118, 121, 3), 2, 0.0), ((118, 121, 3), 2, 0.5), ((118, 121, 1), 4, 0.0), ((118, 121, 1), 4, 0.7),
    ((118, 121, 3), 8, 0.0), ((118, 121, 1), 8, 0.7),          # tiles of one group, few rows and many
    ((260, 263, 1), 16, 0.0), ((260, 263, 1), 16, 0.5),        # larger tiles
    ((34, 37, 3), 32, 0.0), ((34, 37, 3), 32, 1.0), ((60, 52, 3), 16, 0.0),
])
def test_gradients_by_size_and_rows_kept(shape, K, mult):
    """The backward pass samples how many rows its groups keep and takes one kernel or the other."""
    x = synth.add_gaussian_float(synth.clean_image(*shape, 7), 20.0, 7)
    prm = dict(stride=2, window=9, K=K, tau_mult=mult)
    rng = np.random.default_rng(4)
    r = O.denoise(x.astype(np.float64), 20.0, prm, keep_masks=True)
    w = rng.uniform(0.5, 1.5, size=len(r.idx))
    gout = rng.standard_normal(x.shape)
    gx_o, gw_o = O.denoise_fixed_vjp(x.astype(np.float64), gout, r.idx, r.masks, r.U, r.V, w, 8)
    xt, wt = torch.from_numpy(x).cuda(), torch.from_numpy(w.astype(np.float32)).cuda()
    out, info = H.denoise_f32(xt, 20.0, prm, w=wt, return_info=True)
    gx, gw = H.denoise_vjp(xt, 20.0, info["idx"], wt, out, torch.from_numpy(gout.astype(np.float32)).cuda(), prm)
    assert np.abs(gx.cpu().numpy() - gx_o).max() <= 1e-4 * np.abs(gx_o).max()
    assert np.abs(gw.cpu().numpy() - gw_o).max() <= 1e-4 * max(1.0, np.abs(gw_o).max())


@pytest.mark.parametrize("C,K,sizes", [
    (3, 8, [(33, 40), (125, 130), (64, 33), (20, 90), (48, 48)]),              # a larger one among them
    (1, 32, [(40 + i % 7, 41 + i % 5) for i in range(131)]),                   # more than one launch describes
    (3, 16, [(36, 37)] * 2),
    (1, 2, [(8, 8), (9, 31), (8, 60)]),                                        # one reference row
])
def test_small_images_of_a_batch(C, K, sizes):
    """They share their launches: groupings equal those of single calls, pixels to rounding (other filter tiles)."""
    prm = dict(stride=3, window=9, K=K, agg_mode="sparsity" if K == 16 else "uniform")
    sizes = [(h, w) for h, w in sizes if min(9, h - 7) * min(9, w - 7) >= K]
    xs = [torch.from_numpy(synth.add_gaussian(synth.clean_image(h, w, C, 5 + i), 20.0, i)).cuda()
          for i, (h, w) in enumerate(sizes)]
    sig = [10.0 + i % 9 for i in range(len(xs))]
    idx = [torch.empty((H.num_groups(h, w, prm), K), dtype=torch.int32, device="cuda") for h, w in sizes]
    outs = H.denoise_batch(xs, sig, prm, idx_outs=idx)
    again = H.denoise_batch(xs, sig, prm)
    for x, s, o, o2, ix in zip(xs, sig, outs, again, idx):
        want, info = H.denoise(x, s, prm, return_info=True)
        assert torch.equal(ix, info["idx"])
        assert torch.equal(o, o2) and max_abs(o.cpu().numpy(), want.cpu().numpy()) <= PIX_TOL


def test_images_of_a_batch_are_grouped_as_single_ones():
    """Side by side, images take the tensor-core grouping at sizes where one alone does not."""
    prm = dict(stride=3, window=18, K=32)
    xs = [torch.from_numpy(synth.add_gaussian(synth.clean_image(150 + 9 * i, 170, 3, i), 20.0, i)).cuda() for i in range(8)]
    idx = [torch.empty((H.num_groups(*x.shape[:2], prm), 32), dtype=torch.int32, device="cuda") for x in xs]
    outs = H.denoise_batch(xs, [20.0] * 8, prm, idx_outs=idx)
    for x, o, ix in zip(xs, outs, idx):
        want, info = H.denoise(x, 20.0, prm, return_info=True)
        assert torch.equal(ix, info["idx"]) and max_abs(o.cpu().numpy(), want.cpu().numpy()) <= PIX_TOL
