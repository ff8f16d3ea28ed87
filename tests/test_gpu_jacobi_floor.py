"""Eigen-pairs above and in a floor of equal eigenvalues, around the sizes where the
Jacobi kernels change: the separated pairs' residuals in P64, the floor itself in P32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [8, 31, 32, 33, 64, 65, 66, 97, 127, 128, 129, 130, 224, 225, 226, 255, 256])
def test_pairs_above_a_floor(gbpca_lib, B):
    import torch
    rng = np.random.default_rng(B)
    W, _ = np.linalg.qr(rng.standard_normal((B, B)))
    lam = np.full(B, 1e-3)
    lam[:5] = 0.5 ** np.arange(5)
    A = (W * lam) @ W.T
    A = (A + A.T) / 2
    norm = np.linalg.norm(A)
    Ad = torch.from_numpy(A).cuda()

    ev, V, info = (t.cpu().numpy() if hasattr(t, "cpu") else t
                   for t in gbpca_lib.eigh(Ad, precision="p64"))
    assert info["status"] == 0
    # separated pairs: FP64-accurate (1e-13 ||A|| for the products), twice for the difference;
    # their vectors stand clear of all others
    assert np.abs(ev[:5] - lam[:5]).max() <= 1e-12 * norm
    assert np.linalg.norm(A @ V[:, :5] - V[:, :5] * ev[:5], axis=0).max() <= 1e-12 * norm
    assert np.abs(V.T @ V - np.eye(B)).max() <= 1e-12
    assert np.abs(ev[5:] - 1e-3).max() <= 1e-7 * norm

    ev, V, info = (t.cpu().numpy() if hasattr(t, "cpu") else t
                   for t in gbpca_lib.eigh(Ad, precision="p32"))
    assert info["status"] == 0
    # FP32: six roundings of 2^-24 an entry and step, of either sign
    bound = 6 * 2.0 ** -24 * max(info["steps"], 1) ** 0.5 * norm
    assert np.abs(ev - lam).max() <= bound
    assert bound < 0.1 * 1e-3 * norm or B < 6
