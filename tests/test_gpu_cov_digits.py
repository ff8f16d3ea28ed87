"""The P64 covariance from digit products against an extended-precision covariance, at
the edges of its 64-band tiles and 32-pixel chunks, for spectra that need few and many
digits, and for bands without a fixed-point form (which the FP64 products take)."""
import numpy as np
import pytest
import torch

DT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _cube(kind, dtype, N, B, seed):
    r = np.random.default_rng(seed)
    Y = r.uniform(0.0, 1.0, (N, B)) @ np.linalg.qr(r.standard_normal((B, B)))[0]
    if kind == "offset":
        Y += 1000.0 * (1 + np.arange(B))
    elif kind == "wide":            # magnitudes over 2^30 within a band: every digit in use
        Y *= np.exp2(-r.uniform(0, 30, (N, B)))
    elif kind == "scales":          # bands from 2^-40 to 2^40, one constant, one zero
        Y *= np.exp2(np.linspace(-40, 40, B))
        Y[:, 0] = 3.25
        Y[:, B - 1] = 0.0
    elif kind == "outlier":
        Y[N // 2] *= 4096.0
    elif kind == "tiny":            # a spread below the fixed-point scales
        Y[:, 0] *= 1e-37
    return torch.from_numpy(Y.astype(np.float32)).to(DT[dtype])


@pytest.mark.gpu
@pytest.mark.parametrize("kind,dtype,N,B", [
    ("plain", "f32", 2, 2), ("plain", "f32", 31, 63), ("plain", "f32", 33, 64),
    ("plain", "f32", 1000, 65), ("plain", "f32", 1037, 127), ("offset", "f32", 801, 128),
    ("wide", "f32", 1025, 129), ("scales", "f32", 600, 191), ("outlier", "f32", 777, 192),
    ("tiny", "f32", 500, 33), ("plain", "bf16", 700, 200), ("wide", "bf16", 1025, 50),
    ("plain", "f16", 999, 255), ("offset", "f32", 640, 256)])
def test_p64_covariance(gbpca_lib, kind, dtype, N, B):
    Y = _cube(kind, dtype, N, B, seed=N + B)
    mu, C, info = gbpca_lib.covariance(Y.cuda(), "p64")
    X = Y.to(torch.float64).numpy().astype(np.longdouble)
    m = X.mean(0)
    ref = ((X - m).T @ (X - m)) / (N - 1)
    # the sums are taken about the first pixel: a few roundings of 2^-53 of sums that are
    # at most N d_i d_j, d the largest distance from it
    d = np.abs(X - X[0]).max(0)
    err = np.abs(C.cpu().numpy() - ref)
    assert np.all(err <= 16 * 2.0 ** -53 * np.outer(d, d) * N / (N - 1))
    assert np.all(np.abs(mu.cpu().numpy() - m) <= 8 * 2.0 ** -53 * (np.abs(X).max(0) + d))


@pytest.mark.gpu
@pytest.mark.parametrize("value", [float("nan"), -float("nan"), float("inf"), -float("inf")])
def test_p64_covariance_reports_non_finite(gbpca_lib, value):
    Y = _cube("plain", "f32", 300, 70, 5)
    Y[123, 69] = value
    _, _, info = gbpca_lib.covariance(Y.cuda(), "p64")
    assert info["status"] == 3
