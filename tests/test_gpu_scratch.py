"""Calls whose projection planes do not fit: cut into bands of tile rows, or refused, so that the kernels without
planes run. Neither changes a result: the group filter's sums keep their order, and both filters agree bit for bit
(volumes and gradients, whose sums may differ in order, to the bars of the parity tests)."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2508_10307_gb300 as H
from paper_2508_10307_gb300 import _lib, synth
from tests._common import PIX_TOL

pytestmark = pytest.mark.gpu


def _limits(plane_bytes=-1, room=-1):
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    return H.load_library().htsvd_internal_scratch_limits(plane_bytes, room, s)


@pytest.fixture(autouse=True)
def own_workspace():
    H.load_library().htsvd_release_workspace()
    yield
    torch.cuda.synchronize()
    H.load_library().htsvd_release_workspace()


def _counted(call):
    """The call's result and the launches of each kernel in it."""
    _lib.profile_enable(True)
    try:
        res = call()
        torch.cuda.synchronize()
        return res, {k: n for k, (n, _) in _lib.profile_collect(64).items()}
    finally:
        _lib.profile_enable(False)


def _three_ways(call, plane_bytes, planes="planes", per_call=1, bands=3):
    """Results with whole planes, in bands, and without planes; the launches say that each was taken."""
    whole, n = _counted(call)
    assert n.get(planes, 0) == per_call
    _limits(plane_bytes)
    banded, n = _counted(call)
    assert n.get(planes, 0) >= bands * per_call
    H.load_library().htsvd_release_workspace()
    _limits(room=0)
    none, n = _counted(call)
    assert planes not in n
    return whole, banded, none


@pytest.mark.parametrize("shape,prm,sigma", [
    ((124, 131, 3), dict(stride=2, window=11, K=32), 25.0),
    ((131, 124, 3), dict(stride=2, window=9, K=32, tau_mult=1.5), 8.0),       # dense: every band to the tile kernel
    ((131, 124, 1), dict(stride=2, window=9, K=32, tau_mult=2.0, agg_mode="sparsity"), 15.0),
    ((124, 125, 1), dict(stride=2, window=9, K=4, tile=1), 20.0),
])
def test_image(shape, prm, sigma):
    x = torch.from_numpy(synth.add_gaussian(synth.clean_image(*shape, 23), sigma, 23)).cuda()

    def call():
        out, info = H.denoise(x, sigma, prm, return_info=True, masks=True, weights=True)
        return [out, info["idx"], info["masks"], info["weights"]]

    whole, banded, none = _three_ways(call, (1 << 19) * shape[2])
    for a, b, c in zip(whole, banded, none):
        assert torch.equal(a, b) and torch.equal(a, c)


def test_left_over_tiles_of_each_band():
    """Half of the image keeps many coefficients: tiles are left over in some bands, the image as a whole is not."""
    x = synth.add_gaussian(synth.clean_image(150, 151, 3, 29), 4.0, 29)
    rng = np.random.default_rng(3)
    x[90:, :] = rng.integers(0, 256, x[90:, :].shape)
    x = torch.from_numpy(x).cuda()
    whole, banded, none = _three_ways(lambda: [H.denoise(x, 25.0, dict(stride=2, window=9, K=32))], 1 << 21)
    assert torch.equal(whole[0], banded[0]) and torch.equal(whole[0], none[0])


@pytest.mark.parametrize("C,mult", [(3, 0.0), (1, 1.2)])
def test_clip(C, mult):
    clean = synth.clean_image(126, 124, C, 9)
    v = torch.from_numpy(np.stack([synth.add_gaussian(np.roll(clean, t, axis=1), 15.0, 9 + t) for t in range(3)])).cuda()
    whole, banded, none = _three_ways(
        lambda: [H.denoise_video(v, 15.0, dict(stride=2, window=7, K=16, tau_mult=mult), T=1)], 1 << 21, per_call=7)
    assert torch.equal(whole[0], banded[0]) and torch.equal(whole[0], none[0])


@pytest.mark.parametrize("C,K,mult", [(3, 32, 0.0), (1, 16, 1.2)])
def test_gradients(C, K, mult):
    x = torch.from_numpy(synth.add_gaussian_float(synth.clean_image(125, 121, C, 7), 20.0, 7)).cuda()
    prm = dict(stride=2, window=9, K=K, tau_mult=mult)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    out, info = H.denoise_f32(x, 20.0, prm, return_info=True)
    w = 0.5 + torch.rand(info["idx"].shape[0], device="cuda", generator=gen)
    g = torch.randn(x.shape, device="cuda", generator=gen)
    H.load_library().htsvd_release_workspace()
    whole, banded, none = _three_ways(lambda: H.denoise_vjp(x, 20.0, info["idx"], w, out, g, prm), (1 << 20) * C, per_call=2)
    assert torch.equal(whole[0], banded[0])
    for a, b, c in zip(whole, banded, none):      # (the tile kernel adds a weight's gradient with float atomics)
        for r in (b, c):
            assert (a - r).abs().max() <= 1e-4 * max(1.0, a.abs().max().item())


@pytest.mark.parametrize("K,mult", [(32, 0.0), (8, 1.0), (16, 1.0)])
def test_volume(K, mult):
    v = torch.from_numpy(synth.add_gaussian(synth.clean_volume(48, 39, 40, 6), 11.5, 6)).cuda()

    def call():
        out, info = H.denoise_volume(v, 11.5, dict(ps=4, stride=2, window=4, K=K, tau_mult=mult), return_info=True,
                                     masks=True, weights=True)
        return [out, info["masks"], info["weights"]]

    whole, banded, none = _three_ways(call, 6 << 20, planes="volume_planes")
    for r in (banded, none):
        assert torch.equal(whole[1], r[1]) and torch.equal(whole[2], r[2])
        assert (whole[0] - r[0]).abs().max().item() <= PIX_TOL


def test_batch_lane_in_bands():
    prm = dict(stride=2, window=9, K=16)
    xs = [torch.from_numpy(synth.add_gaussian(synth.clean_image(124, 120 + 7 * i, 3, i), 20.0, i)).cuda() for i in range(3)]
    whole = H.denoise_batch(xs, [20.0] * 3, prm)
    torch.cuda.synchronize()
    H.load_library().htsvd_release_workspace()
    _limits(8 << 21)
    banded, n = _counted(lambda: H.denoise_batch(xs, [20.0] * 3, prm))
    assert n["planes"] >= 9
    assert all(torch.equal(a, b) for a, b in zip(whole, banded))


def test_short_of_memory_allocates_once():
    """Where the whole plane finds no room, the band that fitted serves the later calls: none of them allocates
    (each attempt would free it first), and none synchronises."""
    x = torch.from_numpy(synth.add_gaussian(synth.clean_image(330, 331, 3, 3), 20.0, 3)).cuda()
    ref = H.denoise(x, 20.0, dict())
    torch.cuda.synchronize()
    H.load_library().htsvd_release_workspace()
    _limits(room=190 << 20)                      # (129 MB of spilled rows come first, the planes are 90 MB)
    first, n = _counted(lambda: H.denoise(x, 20.0, dict()))
    assert n["planes"] >= 2
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    made = H.load_library().htsvd_internal_scratch_limits(-1, 4 << 20, s)
    for _ in range(3):
        assert torch.equal(H.denoise(x, 20.0, dict()), ref)
    assert H.load_library().htsvd_internal_scratch_limits(-1, -1, s) == made
    assert torch.equal(first, ref)


def test_gradients_at_every_amount_of_room():
    """Whichever buffer of the plane path is the one that finds no room (spilled rows, planes, patch products), the
    call runs without planes."""
    x = torch.from_numpy(synth.add_gaussian_float(synth.clean_image(125, 121, 1, 7), 20.0, 7)).cuda()
    prm = dict(stride=2, window=9, K=16)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    out, info = H.denoise_f32(x, 20.0, prm, return_info=True)
    g = torch.randn(x.shape, device="cuda", generator=gen)
    want = H.denoise_vjp(x, 20.0, info["idx"], None, out, g, prm)

    def at(room):
        torch.cuda.synchronize()
        H.load_library().htsvd_release_workspace()
        _limits(room=room)
        (gx, gw), n = _counted(lambda: H.denoise_vjp(x, 20.0, info["idx"], None, out, g, prm))
        assert (gx - want[0]).abs().max() <= 1e-4 * want[0].abs().max()
        assert (gw - want[1]).abs().max() <= 1e-4 * max(1.0, want[1].abs().max().item())
        return "planes" in n

    lo, hi = 0, 1 << 30
    assert not at(lo) and at(hi)
    while hi - lo > 1 << 12:                     # the least room at which the planes are used, to 4 KB
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if at(mid) else (mid, hi)
    for k in range(12):                          # (the patch products take 54 KB, last of all)
        at(lo - (k << 13))


@pytest.mark.parametrize("batch", [False, True])
def test_planes_are_given_back_before_a_call_fails(batch):
    """A full device: an allocation the call cannot do without fails once, the buffers it can do without are
    freed (the caller's own or those of an earlier batch), and the second attempt succeeds."""
    x = torch.from_numpy(synth.add_gaussian(synth.clean_image(124, 131, 3, 3), 20.0, 3)).cuda()
    y = torch.from_numpy(synth.add_gaussian(synth.clean_image(224, 231, 3, 3), 20.0, 3)).cuda()
    prm = dict(stride=2, window=9, K=16)
    want = H.denoise(y, 20.0, prm)
    torch.cuda.synchronize()
    H.load_library().htsvd_release_workspace()
    H.denoise_batch([x, x], [20.0, 20.0], prm) if batch else H.denoise(x, 20.0, prm)
    torch.cuda.synchronize()
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert H.load_library().htsvd_internal_fail_allocations(1, s) == 0
    assert torch.equal(H.denoise(y, 20.0, prm), want)
    H.load_library().htsvd_internal_fail_allocations(2, s)
    with pytest.raises(_lib.HtsvdError, match="OOM"):
        H.denoise(torch.cat([y, y], 1), 20.0, prm)
    assert torch.equal(H.denoise(y, 20.0, prm), want)
