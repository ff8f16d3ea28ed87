"""The SIMT covariance (P32, P64) at the edges of its tiles and stages: band counts
around the tile and CTA sizes, pixel counts around a stage and a slot, element
types whose rows start between 16-byte units.  Against an FP64 covariance of the
same values; P32 within the bound of FP32 sums of n terms in slots, P64 within
that of FP64 ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [2, 5, 8, 9, 33, 64, 65, 97, 104, 129, 255, 256])
@pytest.mark.parametrize("N,dtype", [(2, "float32"), (15, "bfloat16"), (17, "float16"),
                                     (257, "float32"), (5003, "float16"), (5003, "float32")])
def test_simt_covariance_edges(gbpca_lib, B, N, dtype):
    import torch
    rng = np.random.default_rng(1000 * B + N)
    Y = torch.from_numpy(0.5 + 0.1 * rng.standard_normal((N, B))).to(getattr(torch, dtype)).cuda()
    y = Y.double()
    x = y - y.mean(0)
    C = (x.T @ x) / (N - 1)
    # entry (i, j) is a sum of n products about the first pixel's shift; a slot of at
    # most 256 pixels (here) is summed in the accumulator's type
    d = y - y[0]
    size = (d.abs().T @ d.abs()) / (N - 1)
    m = min(N, 256) + 2
    for prec, u in (("p32", 2.0 ** -24), ("p64", 2.0 ** -53)):
        mu, cov, info = gbpca_lib.covariance(Y, prec)
        assert info["status"] == 0
        bound = 2 * m * u * size + 64 * 2.0 ** -53 * size
        assert bool(((cov - C).abs() <= bound).all()), (B, N, dtype, prec)
        assert bool(((mu - y.mean(0)).abs() <= 64 * 2.0 ** (-24 if prec == "p32" else -52)
                     * (d.abs().mean(0) + 1e-9 * (prec == "p32")) + 4e-16).all())
