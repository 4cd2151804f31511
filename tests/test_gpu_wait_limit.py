"""Waits for the tensor cores that run out (by a switch of the stream's workspace): the call's groups hold positions inside
the image, the status comes once, from the next call or from the call itself where it waits for the device, and
the call after it groups as ever. Images of at least 76 tiles of 128 references, which the tensor cores group."""
import ctypes

import numpy as np
import pytest
import torch

import paper_2508_10307_gb300 as H
from oracle import htsvd_oracle as O
from paper_2508_10307_gb300 import _lib, synth

pytestmark = pytest.mark.gpu

PRM = dict(stride=3, window=18, K=32)


def _give_up(on):
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert H.load_library().htsvd_internal_give_up_waits(on, s) == 0


@pytest.fixture
def no_waiting():
    _give_up(1)
    yield
    _give_up(0)


def _noisy(C, seed=3):
    return torch.from_numpy(synth.add_gaussian(synth.clean_image(330, 331, C, seed), 20.0, seed)).cuda()


@pytest.mark.parametrize("C", [1, 3])
def test_status_comes_once_and_indices_stay_inside(C, no_waiting):
    x = _noisy(C)
    out, info = H.denoise(x, 20.0, PRM, return_info=True)
    torch.cuda.synchronize()
    idx = info["idx"].cpu().numpy()
    y, xx = idx // 331, idx % 331
    assert idx.min() >= 0 and y.max() <= 330 - 8 and xx.max() <= 331 - 8
    rows, cols = O.reference_positions(330, 8, 3), O.reference_positions(331, 8, 3)
    assert np.array_equal(idx[:, 0], (np.asarray(rows)[:, None] * 331 + np.asarray(cols)[None, :]).ravel())
    _give_up(0)
    with pytest.raises(_lib.HtsvdError, match="TIMEOUT"):
        H.denoise(x, 20.0, PRM)
    ref, good = H.denoise(x, 20.0, PRM, return_info=True)
    with torch.cuda.stream(torch.cuda.Stream()):
        again, other = H.denoise(x, 20.0, PRM, return_info=True)
        torch.cuda.synchronize()
    assert torch.equal(good["idx"], other["idx"]) and torch.equal(ref, again)


def test_a_call_that_waits_for_the_device_reports_its_own(no_waiting):
    x = _noisy(3)
    with pytest.raises(_lib.HtsvdError, match="TIMEOUT"):
        H.denoise(x, 20.0, PRM, basis_gap=True, return_info=True)
    _give_up(0)
    H.denoise(x, 20.0, PRM, basis_gap=True, return_info=True)


def test_a_batch_reports_the_lanes_of_the_one_before(no_waiting):
    xs = [_noisy(3, 3 + i) for i in range(3)]
    H.denoise_batch(xs, [20.0] * 3, PRM)
    torch.cuda.synchronize()
    _give_up(0)
    with pytest.raises(_lib.HtsvdError, match="TIMEOUT"):
        H.denoise_batch(xs[:1], [20.0], PRM)         # (one lane: the others' words count as well)
    for x, o in zip(xs, H.denoise_batch(xs, [20.0] * 3, PRM)):
        assert (o - H.denoise(x, 20.0, PRM)).abs().max().item() <= 1e-3
