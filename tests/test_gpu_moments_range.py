"""The weighted covariance of FP32 samplers where 32-bit floating point would
run out of range or of bits.

Its products and sums are pairs of FP32 values at scales taken from a block's
first rows and largest weight.  Where those do not suffice the block must fall
back to FP64: values far larger or smaller than the first rows', and a block
whose heaviest particle contributes nothing.  And the pairs themselves must
carry about twice FP32's digits: a plain FP32 product or sum does not pass."""
import numpy as np
import pytest
import torch

from paper_1905_10252_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_1905_10252_gb300 import build, native

    build.build()
    native.lib()
    return native


def _sampler(nat, n, d, seed=3):
    mu, sigma = inputs.gaussian_target(d, seed=seed)
    return nat.Sampler(n, d, dtype=torch.float32, seed=seed + n, mu=mu, sigma=sigma, step=0.25, init_scale=1.5)


def _weights(S):
    st = S.stats()
    return torch.exp(S.logw - st["max_logw"]) / np.exp(st["lse"] - st["max_logw"])


def _compare(S, mean, cov, r, eps):
    """Entry by entry: |cov - sum w r r| <= eps sum w |r r|, r FP64 values."""
    w = _weights(S)
    ref = torch.einsum("i,ia,ib->ab", w, r, r)
    mag = torch.einsum("i,ia,ib->ab", w, r.abs(), r.abs())
    assert bool(torch.isfinite(mag).all()) and bool(torch.isfinite(cov).all())
    err = (cov - ref).abs()
    assert bool((err <= eps * mag + 1e-300).all()), float((err / (eps * mag + 1e-300)).max())
    assert torch.equal(cov, cov.T)


# two factors of 2^-24 (the rows' differences rounded to FP32), with a margin of 1/2
ROW_EPS = 1.5 * 2.0**-23


@pytest.mark.parametrize("n,d", [(300, 3), (5003, 16), (20011, 32), (300007, 9)])
@pytest.mark.parametrize("far", [1e13, 1e25])
def test_rows_far_larger_than_the_first(nat, n, d, far):
    S = _sampler(nat, n, d)
    S.move()
    S.reweight()
    mean = S.estimate()[0]
    x = S.current()[0]
    x[:64] = (mean + 1e-6 * (x[:64].double() - mean)).float()
    x[100::71, d // 2] *= far
    x[n - 1] = -far
    mean2, cov = S.estimate(cov=True)
    assert torch.equal(mean, mean2)
    _compare(S, mean, cov, S.current()[0].double() - mean, ROW_EPS)


@pytest.mark.parametrize("n,d", [(300, 3), (5003, 16), (20011, 32)])
@pytest.mark.parametrize("far", [1e14, 1e30])
def test_rows_far_smaller_than_the_first(nat, n, d, far):
    S = _sampler(nat, n, d)
    S.move()
    S.reweight()
    mean = S.estimate()[0]
    S.current()[0][7] = far  # one of the rows that give the scale, with weight zero
    S.logw[7] = -np.inf
    cov = S.estimate(cov=True)[1]
    _compare(S, mean, cov, S.current()[0].double() - mean, ROW_EPS)


@pytest.mark.parametrize("gap", [70.0, 90.0, 250.0, 600.0])
@pytest.mark.parametrize("n,d", [(100, 4), (3000, 17)])
def test_heaviest_particle_at_the_mean(nat, n, d, gap):
    """One particle with all the weight that the 62 bits of eq. (7) hold: the
    mean is that particle, and the covariance is what the others add."""
    S = _sampler(nat, n, d)
    S.move()
    S.reweight()
    S.logw.copy_(torch.randn(n, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1)))
    S.logw[5] = gap + 8.0
    S.reweight()  # (log pi is unchanged: so is log w)
    mean, cov = S.estimate(cov=True)
    x = S.current()[0].double()
    assert torch.equal(mean, x[5])
    assert float(cov.diagonal().min()) > 0.0
    _compare(S, mean, cov, x - mean, ROW_EPS)


@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_non_finite_row_reaches_its_column(nat, value):
    S = _sampler(nat, 5003, 6)
    S.move()
    S.reweight()
    S.current()[0][4000, 2] = value
    cov = S.estimate(cov=True)[1]
    hit = torch.zeros(6, 6, dtype=torch.bool, device="cuda")
    hit[2, :] = hit[:, 2] = True
    assert not bool(torch.isfinite(cov[hit]).any()) and bool(torch.isfinite(cov[~hit]).all())


def _centred(x, mean):
    """The rows' differences in FP32, as the kernel rounds them (32-bit operations one by one)."""
    x = x.cpu().numpy()
    m = mean.cpu().numpy()
    mh = m.astype(np.float32)
    ml = (m - mh.astype(np.float64)).astype(np.float32)
    d = x - mh
    b = d - x
    e = (x - (d - b)) - (mh + b)
    r = d + (e - ml)
    assert r.dtype == np.float32
    return torch.from_numpy(r).double().cuda()


@pytest.mark.parametrize("n,d", [(1, 1), (255, 2), (1000, 4), (1500, 8), (2500, 12), (3001, 16), (4000, 20), (5003, 32)])
def test_pairs_carry_twice_the_digits(nat, n, d):
    """Against FP64 sums over the same FP32 differences.  Relative to the terms'
    magnitudes: the weight 2^-45, its product with a difference and that
    product's 2^-46 each; and the low words of a sum of k rows (k <= 32 at these
    sizes) at most k roundings of a value up to k 2^-24 of it, k^2 2^-48 =
    2^-38.  FP32 products or sums alone would be off by 2^-24."""
    S = _sampler(nat, n, d)
    S.move()
    S.reweight()
    mean, cov = S.estimate(cov=True)
    _compare(S, mean, cov, _centred(S.current()[0], mean), 2.0**-37)
