"""P64 band means and covariance of large cubes with outlying pixels (hot, saturated
and no-data values) against extended precision, relative to the variances."""
import numpy as np
import pytest
import torch


def _moments(Y):
    """Band means, covariance and the sums of squares about the first pixel, in extended
    precision with pairwise sums."""
    N, B = Y.shape
    X = [Y[:, b].astype(np.longdouble) - np.longdouble(Y[0, b]) for b in range(B)]
    d = np.array([x.sum() / N for x in X])
    S2 = np.array([[(X[i] * X[j]).sum() for j in range(B)] for i in range(B)])
    return Y[0].astype(np.longdouble) + d, (S2 - N * np.outer(d, d)) / (N - 1), np.diag(S2)


def _check(cov, Y):
    mu, C, info = cov
    N = Y.shape[0]
    m, ref, sq = _moments(Y)
    # at most 320 partial sums, added by eight warps; every running sum is at most
    # sqrt(S2_aa S2_bb): 320 / 8 + 8 roundings, and sixteen for the partials, the last
    # subtraction of N d_a d_b, the quotient
    bound = (320 / 8 + 8 + 16) * 2.0 ** -53 * np.sqrt(np.outer(sq, sq)) / (N - 1)
    assert info["status"] == 0
    assert np.all(np.abs(C.cpu().numpy() - ref) <= bound)
    assert np.all(np.abs(mu.cpu().numpy() - m) <= 64 * 2.0 ** -53 * (np.abs(m) + np.sqrt(sq / N)))


@pytest.mark.gpu
@pytest.mark.parametrize("N", [100_000, 1_000_000])
@pytest.mark.parametrize("value", [300.0, 1000.0, 9999.0, -9999.0, 65535.0])
def test_p64_covariance_with_one_outlying_pixel(gbpca_lib, N, value):
    r = np.random.default_rng(N)
    Y = r.uniform(0.0, 1.0, (N, 3)).astype(np.float32)
    Y[0] = 0.5
    Y[N // 3, 0] = value                # band 0 alone
    Y[N // 2, :2] = value               # bands 0 and 1 at one pixel
    _check(gbpca_lib.covariance(torch.from_numpy(Y).cuda(), "p64"), Y)


@pytest.mark.gpu
def test_p64_covariance_with_outliers_in_every_chunk(gbpca_lib):
    """Values over 2^13 in magnitude within every 32 pixels: all levels of the products."""
    N = 65_536
    r = np.random.default_rng(1)
    Y = (r.uniform(0.0, 1.0, (N, 3)) * np.exp2(r.integers(-13, 1, (N, 3)))).astype(np.float32)
    Y[0] = 0.25
    _check(gbpca_lib.covariance(torch.from_numpy(Y).cuda(), "p64"), Y)
