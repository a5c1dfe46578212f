"""The tensor-core likelihood at values without a finite log-target: a NaN or
infinite coordinate is reported; a particle so far out that the sum of |z|
leaves FP32 has log pi = -inf and weight zero, and one whose sums only leave
FP32 in the total keeps its finite log pi."""
import numpy as np
import pytest
import torch

from paper_1905_10252_gb300 import inputs

pytestmark = pytest.mark.gpu

N, D, M = 1000, 5, 700


@pytest.fixture(scope="module")
def nat():
    from paper_1905_10252_gb300 import build, native

    build.build()
    native.lib()
    return native


def _sampler(nat, n=N, d=D, m=M, X=None, y=None):
    if X is None:
        X, y, _ = inputs.logistic_data(m, d, seed=3)
    return nat.Sampler(n, d, dtype=torch.float32, seed=5, target="logistic", X=X, y=y, prior_var=4.0, step=0.2,
                       resample_mode=nat.RESAMPLE_NEVER)


# the NaN of the GPU's arithmetic (whose BF16 images are zero), other NaNs, the infinities
BITS = [0x7FFFFFFF, 0x7FC00000, 0x7F800001, -1, 0x7F800000, -0x800000]


@pytest.mark.parametrize("call", ["reweight", "step"])
@pytest.mark.parametrize("bits", BITS)
@pytest.mark.parametrize("row,col", [(0, 0), (131, 4), (999, 2)])
def test_non_finite_coordinate_is_reported(nat, bits, row, col, call):
    S = _sampler(nat)
    S.sync()
    S.current()[0].view(torch.int32)[row, col] = bits
    S.reweight() if call == "reweight" else S.step(1)
    with pytest.raises(nat.SmcError) as e:
        S.sync()
    assert e.value.code == nat.SMC_ENONFINITE
    S.close()


@pytest.mark.parametrize("call", ["reweight", "step"])
@pytest.mark.parametrize("value", [3e36, -3e36])
@pytest.mark.parametrize("m", [200, 700, 4097])
def test_overflowing_sum_is_weight_zero(nat, m, value, call):
    # |z| up to 1e37, its sum over a few hundred rows beyond 3.4e38
    S = _sampler(nat, m=m)
    S.sync()
    S.current()[0][[3, 500], 1] = value
    mean = S.step(1)["mean"] if call == "step" else (S.reweight(), S.estimate()[0])[1]
    S.sync()
    lp, lw = S.current()[1], S.logw
    out = torch.zeros(N, dtype=torch.bool, device="cuda")
    out[[3, 500]] = True
    assert bool((lp[out] == -np.inf).all()) and bool((lw[out] == -np.inf).all())
    assert bool(torch.isfinite(lp[~out]).all()) and bool(torch.isfinite(lw[~out]).all())
    assert bool(torch.isfinite(mean).all())
    S.close()


def test_total_beyond_fp32_of_finite_partial_sums(nat):
    """z = 2^118 in each of 8192 rows: 2^127.5 over the 512 rows of a partial
    sum, 2^131 in all, against b.X^T(y - 1/2) = 2^130, so that log pi is the
    prior's -2^113 and the rounding of z.  Per row 2^-16 |z| (the products'
    split) and 512 2^-24 of the partial sum (FP32): |log pi| <= 2^113 +
    2^130 (2^-16 + 2^-15) < 2^117."""
    m = 8192
    X, y = np.full((m, 1), 2.0**60, np.float32), np.ones(m, np.float32)
    S = _sampler(nat, n=300, d=1, X=X, y=y)
    S.sync()
    S.current()[0][7, 0] = 2.0**58
    S.reweight()
    S.sync()
    lp = float(S.current()[1][7])
    assert np.isfinite(lp) and abs(lp) < 2.0**117, lp
    assert np.isfinite(float(S.logw[7]))
    S.close()
