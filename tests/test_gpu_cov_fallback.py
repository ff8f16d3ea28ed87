"""The FP64 sums behind the digit products of a P64 covariance: a band without a
fixed-point form gives the sums of a fit, slot by slot, and a workspace sized for more
bands serves fewer."""
import numpy as np
import pytest
import torch


@pytest.mark.gpu
@pytest.mark.parametrize("N,B", [(3001, 17), (20_003, 60), (100_000, 256)])
def test_fallback_sums_in_the_slots_of_a_fit(gbpca_lib, N, B):
    Y = np.random.default_rng(B).uniform(0.0, 1.0, (N, B)).astype(np.float32)
    Y[:, 3] *= np.float32(1e-37)       # no fixed-point scale: every band takes the FP64 sums
    Yd = torch.from_numpy(Y).cuda()
    mu, C, info = gbpca_lib.covariance(Yd, "p64")
    fit = gbpca_lib.fit(Yd, 1, precision="p64", project=False)
    assert info["status"] == 0
    assert torch.equal(mu, fit[0])
    lam = torch.linalg.eigvalsh(C).flip(0)
    assert abs(lam[0].item() - fit[1][0].item()) <= 1e-12 * lam[0].item()


@pytest.mark.gpu
def test_workspace_of_more_bands_serves_fewer(gbpca_lib):
    g = gbpca_lib
    N = 100_000
    ws = g.make_workspace(N, 100, 4, 0, "p64", torch.device("cuda"))
    for B in (100, 63, 40):
        Y = torch.rand(N, B, device="cuda")
        _, C, info = g.covariance(Y, "p64", workspace=ws)
        assert info["status"] == 0
        ev = g.fit(Y, 4, precision="p64", workspace=ws)[1]
        ref = torch.linalg.eigvalsh(C).flip(0)
        assert (ev - ref).abs().max().item() <= 1e-10 * ref[0].item()


@pytest.mark.gpu
def test_constant_bands_of_every_size(gbpca_lib):
    """A band of one value has a fixed-point form whatever the value (a fill value of 1e37 and
    beyond as well): zero covariances, the value as its mean."""
    values = (0.0, 3.25, -1e37, 9.96921e36, 3.4e38, 2.0 ** 63, 1e-30, -1e-39)
    Y = np.random.default_rng(2).uniform(0.0, 1.0, (5000, len(values) + 2)).astype(np.float32)
    Y[:, :len(values)] = values
    mu, C, info = gbpca_lib.covariance(torch.from_numpy(Y).cuda(), "p64")
    assert info["status"] == 0
    assert np.array_equal(mu.cpu().numpy()[:len(values)], Y[0, :len(values)].astype(np.float64))
    assert not C[:len(values)].any()
    ref = np.cov(Y[:, len(values):].astype(np.float64).T)
    assert np.abs(C[len(values):, len(values):].cpu().numpy() - ref).max() <= 1e-14


@pytest.mark.gpu
@pytest.mark.parametrize("kind,fallback", [("plain", 0), ("no-data pixel", 0), ("constant band", 0),
                                           ("tiny spread", 1), ("fill value", 1), ("infinity", 1)])
def test_p64_covariance_reports_its_form(gbpca_lib, kind, fallback):
    Y = np.random.default_rng(3).uniform(0.0, 1.0, (50_000, 40)).astype(np.float32)
    if kind == "no-data pixel":
        Y[123] = -9999.0
    elif kind == "constant band":
        Y[:, 7] = 9.96921e36
    elif kind == "tiny spread":
        Y[:, 7] *= np.float32(1e-30)
    elif kind == "fill value":
        Y[123] = 9.96921e36
    elif kind == "infinity":
        Y[123, 7] = np.inf
    _, _, info = gbpca_lib.covariance(torch.from_numpy(Y).cuda(), "p64")
    assert info["status"] == (3 if kind == "infinity" else 0)
    assert info["cov_fallback"] == fallback
    # a fit adds in FP64 by itself
    assert gbpca_lib.fit(torch.from_numpy(Y).cuda(), 1, precision="p64")[4]["cov_fallback"] == 0
