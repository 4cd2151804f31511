"""Bases of the device eigensolver (FP32 sweeps, then FP64 ones) against the FP64 oracle's, over numbers of
references from a few to several chunks of the moment kernel, and over scales of the image. Bar as in the
parity tests: 1e-9."""
import numpy as np
import pytest
import torch

import paper_2508_10307_gb300 as H
from oracle import htsvd_oracle as O
from paper_2508_10307_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["natural", "faint", "saturated"])
@pytest.mark.parametrize("shape", [(17, 21, 3), (40, 33, 1), (64, 70, 3), (151, 330, 3), (255, 131, 1)])
def test_device_bases_match_oracle(shape, kind):
    x = synth.add_gaussian(synth.clean_image(*shape, 19), 20.0, 19)
    if kind == "faint":                      # eigenvalues near the noise floor of small integers
        x = (x >> 5).astype(np.uint8)
    elif kind == "saturated":
        x = np.where(x > 127, 255, x & 3).astype(np.uint8)
    prm = dict(stride=3, window=7, K=4)
    _, info = H.denoise(torch.from_numpy(x).cuda(), 10.0, prm, return_info=True, basis=True)
    b = info["basis"].cpu().numpy()
    z = b[..., 0] + 1j * b[..., 1]
    U, V, _, _ = O.global_basis(O.reference_patches(x, O.Params.of(prm)))
    assert np.abs(z[0] - U).max() < 1e-9 and np.abs(z[1] - V).max() < 1e-9
