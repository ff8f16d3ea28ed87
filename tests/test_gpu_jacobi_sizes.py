"""The Jacobi kernels around the sizes where their work lists, V widths and the
choice between them change: eigen-pairs of matrices with a decaying and with a
clustered spectrum against FP64, even and odd orders."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _matrix(B, kind, rng):
    W, _ = np.linalg.qr(rng.standard_normal((B, B)))
    lam = np.exp(-np.linspace(0.0, 6.0, B)) if kind == "decaying" else np.full(B, 1e-3)
    if kind == "clustered":
        lam[: min(B, 5)] = 0.5 ** np.arange(min(B, 5))
    A = (W * lam) @ W.T
    return (A + A.T) / 2


@pytest.mark.parametrize("kind", ["decaying", "clustered"])
@pytest.mark.parametrize("B", [2, 3, 4, 5, 30, 31, 32, 33, 62, 63, 64, 65, 66, 67, 96, 97, 126, 127,
                               128, 129, 130, 255, 256])
def test_eigenpairs_at_size_edges(gbpca_lib, B, kind):
    import torch
    A = _matrix(B, kind, np.random.default_rng(B))
    norm = np.linalg.norm(A)
    ref = np.sort(np.linalg.eigvalsh(A))[::-1]
    Ad = torch.from_numpy(A).cuda()
    for prec in ("p32", "p64"):
        lam, V, info = gbpca_lib.eigh(Ad, precision=prec)
        assert info["status"] == 0
        lam, V = lam.cpu().numpy(), V.cpu().numpy()
        # FP32: every step turns each entry and each row of V once, with at most six
        # roundings of 2^-24; P64: the refined pairs
        bound = 6 * 2.0 ** -24 * max(info["steps"], 1) if prec == "p32" else 1e-10
        assert np.abs(lam - ref).max() <= bound * norm, (B, kind, prec)
        assert np.abs(V.T @ V - np.eye(B)).max() <= bound * B ** 0.5, (B, kind, prec)
        if prec == "p32" or kind == "decaying":
            assert np.linalg.norm(A @ V - V * lam) <= 2 * bound * norm * B ** 0.5, (B, kind, prec)
