"""The FP64 SIMT covariance at the edges of its tiles and stages: behind the digit
products of a P64 covariance call (one band with a spread below their scales sends the
cube there) and as a P64 fit runs it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(2, "float32"), (15, "bfloat16"), (17, "float16"), (257, "float32"),
         (5003, "float16"), (5003, "float32"), (82_001, "bfloat16")]
BANDS = [2, 5, 8, 9, 33, 64, 65, 97, 104, 129, 255, 256]


def _cube(N, B, dtype, tiny):
    import torch
    rng = np.random.default_rng(1000 * B + N)
    Y = torch.from_numpy(0.5 + 0.1 * rng.standard_normal((N, B))).to(getattr(torch, dtype)).cuda()
    if tiny:
        Y[:, B - 1] *= 2.0 ** -110 if dtype != "float16" else 0.0
    return Y


@pytest.mark.parametrize("B", BANDS)
@pytest.mark.parametrize("N,dtype", [s for s in SIZES if s[1] != "float16"])
def test_fp64_sums_behind_the_digit_products(gbpca_lib, B, N, dtype):
    Y = _cube(N, B, dtype, tiny=True)
    mu, cov, info = gbpca_lib.covariance(Y, "p64")
    assert info["status"] == 0 and info["cov_fallback"] == 1
    y = Y.double()
    x = y - y.mean(0)
    C = (x.T @ x) / (N - 1)
    # sums of at most 257 products about the first pixel in each of at most 320 slots,
    # and the reference's own sums of N products
    d = (y - y[0]).abs()
    size = (d.T @ d) / (N - 1)
    bound = (2 * min(N, 257) + 64 + 4 * N ** 0.5) * 2.0 ** -53 * size
    assert bool(((cov - C).abs() <= bound).all())
    assert bool(((mu - y.mean(0)).abs() <= 64 * 2.0 ** -52 * (d.mean(0) + y.abs().mean(0))).all())


@pytest.mark.parametrize("B", BANDS)
@pytest.mark.parametrize("N,dtype", SIZES)
def test_fit_of_every_shape(gbpca_lib, B, N, dtype):
    """The eigen-pairs of a P64 fit put together again: 1e-7 ||C|| for each pair at least."""
    import torch
    Y = _cube(N, B, dtype, tiny=False)
    mu, ev, V, _, info = gbpca_lib.fit(Y, 1, precision="p64", project=False)
    assert info["status"] == 0
    y = Y.double()
    x = y - y.mean(0)
    C = (x.T @ x) / (N - 1)
    norm = torch.linalg.norm(C)
    assert torch.linalg.norm((V * ev) @ V.T - C) <= 1e-7 * B ** 0.5 * norm
    assert (ev.sum() - C.trace()).abs() <= 1e-7 * B * norm
    assert bool(((mu - y.mean(0)).abs() <= 64 * 2.0 ** -52 * y.abs().mean(0)).all())
