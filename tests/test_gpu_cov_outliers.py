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


@pytest.mark.gpu
@pytest.mark.parametrize("big", [2.0 ** 30, 2.0 ** 45, 2.0 ** 54, 9.96921e36])
def test_p64_covariance_far_below_an_outlier(gbpca_lib, big):
    """One fill value in band 0, where band 1 equals the shift: their covariance is that
    of the other pixels, each entry to FP64."""
    N = 8192
    r = np.random.default_rng(7)
    half = r.uniform(0.0, 0.25, (N // 2 - 1, 2)).astype(np.float32)
    half[:, 1] = half[:, 0] * np.float32(0.5)
    Y = np.full((N, 2), 0.5, dtype=np.float32)
    Y[1:N // 2] += half                 # band 1's values are symmetric about the shift:
    Y[N // 2:N - 1] = 1.0 - Y[1:N // 2]   # its mean is the shift, so nothing cancels
    Y[N - 1, 0] = big
    _, C, info = gbpca_lib.covariance(torch.from_numpy(Y).cuda(), "p64")
    X = Y.astype(np.longdouble) - np.longdouble(0.5)
    assert info["status"] == 0 and X[:, 1].sum() == 0
    # FP64 sums of N terms (32 slots of 256 pixels)
    bound = (256 + 32) * 2.0 ** -53 * (np.abs(X[:, 0]) * np.abs(X[:, 1])).sum() / (N - 1)
    assert abs(np.longdouble(C[0, 1].item()) - (X[:, 0] * X[:, 1]).sum() / (N - 1)) <= bound


@pytest.mark.gpu
@pytest.mark.parametrize("count", [3, 16, 17, 200])
def test_p64_covariance_with_values_near_zero(gbpca_lib, count):
    """A few values, or more than are let pass, with bits below the fixed point's unit."""
    N = 40_000
    r = np.random.default_rng(count)
    Y = r.uniform(0.5, 1.0, (N, 3)).astype(np.float32)
    Y[0] = 0.75
    Y[7] = 60_000.0
    Y[r.permutation(np.arange(8, N))[:count], 1] = r.uniform(1e-9, 1e-6, count)
    mu, C, info = gbpca_lib.covariance(torch.from_numpy(Y).cuda(), "p64")
    m, ref, sq = _moments(Y)
    # FP64 sums of 256 pixels beside the roundings of _check, and 2^-52 sqrt(2 x 16)
    bound = (256 + 64 + 12) * 2.0 ** -53 * np.sqrt(np.outer(sq, sq)) / (N - 1)
    assert info["status"] == 0
    assert np.all(np.abs(C.cpu().numpy() - ref) <= bound)
