"""Bases of images whose eigenvalues lie close together: the device solver's FP32 start must leave nothing behind.
A basis is orthonormal to rounding and diagonalises the exact scatter matrix to 1e-13 of its largest eigenvalue and
the rounding with which the matrix is formed (a slice's entries are differences of moments, whose scale is the largest
eigenvalue of all slices: 8 eps of that); where the gap allows it, it equals the FP64 oracle's to the bound of a
perturbation of that size."""
import numpy as np
import pytest
import torch

import paper_2508_10307_gb300 as H
from oracle import htsvd_oracle as O

pytestmark = pytest.mark.gpu


def _image(kind, C, rng):
    n = 96
    if kind == "noise":                          # seven nearly equal eigenvalues under the mean's
        x = rng.normal(128, 20, (n, n, C))
    elif kind == "faint":                        # the same a million times smaller than the mean's
        x = 200.0 + (rng.random((n, n, C)) < 0.01)
    elif kind == "symmetric":                    # mirrored rows: pairs of eigenvectors even and odd
        x = rng.normal(128, 30, (n, n, C))
        x = (x + x[::-1]) / 2
    else:                                        # channels nearly equal: the first slice a million times smaller
        x = np.repeat(rng.normal(128, 30, (n, n, 1)), C, 2) + (rng.random((n, n, C)) < 0.02)
    return np.clip(np.rint(x), 0, 255).astype(np.uint8)


@pytest.mark.parametrize("C", [1, 3])
@pytest.mark.parametrize("kind", ["noise", "faint", "symmetric", "channels"])
def test_close_eigenvalues(kind, C):
    x = _image(kind, C, np.random.default_rng(8))
    prm = dict(stride=3, window=7, K=4)
    _, info = H.denoise(torch.from_numpy(x).cuda(), 10.0, prm, return_info=True, basis=True)
    b = info["basis"].cpu().numpy()
    z = b[..., 0] + 1j * b[..., 1]
    P = O.reference_patches(x, O.Params.of(prm))
    X = np.fft.fft(P.astype(np.float64), axis=-1)
    want = O.global_basis(P)
    top = max(want[2].max(), want[3].max())
    for f in range(C // 2 + 1):
        r = X[..., f].transpose(1, 0, 2).reshape(8, -1)
        k = X[..., f].transpose(2, 0, 1).reshape(8, -1)
        for which, A in ((0, r @ r.conj().T), (1, k.conj() @ k.T)):
            V = z[which, f]
            assert np.abs(V.conj().T @ V - np.eye(8)).max() < 1e-13
            D = V.conj().T @ A @ V
            lam = np.linalg.eigvalsh(A)[::-1]
            lim = 1e-13 * lam[0] + 8 * np.finfo(float).eps * top
            assert np.abs(D - np.diag(np.diag(D))).max() <= lim
            gap = np.diff(-lam) / lam[0]
            for i in range(8):
                g = min(gap[max(i - 1, 0)], gap[min(i, 6)])
                if g > 1e-9:
                    assert np.abs(V[:, i] - want[which][f][:, i]).max() <= max(1e-9, lim / lam[0] / g)
