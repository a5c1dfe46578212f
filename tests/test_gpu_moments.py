"""The weighted covariance of the estimate (eq. (7)) against 64-bit sums over
the same particles and weights."""
import numpy as np
import pytest
import torch

from paper_1905_10252_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_1905_10252_gb300 import native

    native.lib()
    return native


def _sampler(nat, n, d, dtype, scale=1.0, seed=3):
    mu, sigma = inputs.gaussian_target(d, seed=seed)
    # columns of very different magnitude when scale != 1
    s = np.array([scale ** (c % 3) for c in range(d)])
    return nat.Sampler(n, d, dtype=dtype, seed=seed + n, mu=mu * s, sigma=sigma * np.outer(s, s), step=0.25,
                       init_scale=1.5)


def _check(nat, S, mean, cov, dtype):
    """|cov - ref| entry by entry within the rounding of the rows' differences
    to the particle precision (two factors of 2^-24, or FP64's sums) times the
    sum of the terms' magnitudes; each FP64 weight itself is good to 2^-50."""
    x = S.current()[0].double()
    st = S.stats()
    S.sync()
    lw = S.logw
    w = torch.exp(lw - st["max_logw"]) / np.exp(st["lse"] - st["max_logw"])
    r = x - mean
    ref = torch.einsum("i,ia,ib->ab", w, r, r)
    mag = torch.einsum("i,ia,ib->ab", w, r.abs(), r.abs())
    eps = 2.0**-23 if dtype == torch.float32 else 2.0**-44
    # the difference itself: the mean's FP64 rounding against a particle
    bound = eps * 1.5 * mag + 1e-300
    err = (cov - ref).abs()
    assert bool((err <= bound).all()), float((err / bound).max())
    assert torch.equal(cov, cov.T)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n,d", [(1, 1), (7, 3), (63, 2), (255, 4), (257, 5), (1000, 8), (4097, 12), (5003, 16),
                                 (20011, 17), (9001, 25), (3001, 31), (50021, 32), (300007, 9)])
def test_covariance_shapes(nat, n, d, dtype):
    S = _sampler(nat, n, d, dtype)
    S.move()
    S.reweight()
    mean, cov = S.estimate(cov=True)
    _check(nat, S, mean, cov, dtype)


@pytest.mark.parametrize("scale", [1e-9, 1e7])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_covariance_columns_of_different_magnitude(nat, scale, dtype):
    S = _sampler(nat, 3000, 7, dtype, scale=scale)
    S.move()
    S.reweight()
    # settle on the target: the weights stay those of this reweight
    mean, cov = S.estimate(cov=True)
    _check(nat, S, mean, cov, dtype)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_covariance_after_a_reset_of_the_weights(nat, dtype):
    """estimate() after a redistribution: log w is -log N, above or below the
    last reweight's maximum."""
    S = _sampler(nat, 6007, 6, dtype)
    S.move()
    S.reweight()
    nc, _ = S.resample()
    S.redistribute(nc)
    mean, cov = S.estimate(cov=True)
    _check(nat, S, mean, cov, dtype)


@pytest.mark.parametrize("gap", [0.0, 30.0, 60.0, 200.0, 900.0])
def test_covariance_of_far_apart_weights(nat, gap):
    """Weights given by the caller: two groups whose log-weights differ by
    `gap`, the heavy group a single particle, and -inf entries."""
    n, d = 2048, 5
    S = _sampler(nat, n, d, torch.float32)
    S.move()
    S.reweight()
    mean, _ = S.estimate()
    st = S.stats()
    lw = torch.full((n,), st["max_logw"] - gap, dtype=torch.float64, device="cuda")
    lw[5] = st["max_logw"]
    lw[100:200] = -np.inf
    S.logw.copy_(lw)
    mean2, cov = S.estimate(cov=True)
    assert torch.equal(mean, mean2)
    _check(nat, S, mean, cov, torch.float32)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_nan_weight_reaches_the_covariance(nat, dtype):
    S = _sampler(nat, 700, 5, dtype)
    S.move()
    S.reweight()
    S.logw[123] = float("nan")
    _, cov = S.estimate(cov=True)
    assert bool(torch.isnan(cov).all())
