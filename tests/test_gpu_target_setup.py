"""A covariance that is not positive definite is reported whichever column shows
it, and one that is becomes the sampler's factor: every warp of the set-up
leaves at the same column."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_1905_10252_gb300 import build, native

    build.build()
    native.lib()
    return native


def _sigma(d, seed=0):
    a = np.random.default_rng(seed + d).standard_normal((d, d + 2))
    return a @ a.T + 0.1 * np.eye(d)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("d", [1, 2, 4, 5, 8, 13, 16, 17, 31, 32])
def test_each_column_of_an_indefinite_covariance(nat, d, dtype):
    good = nat.Sampler(100, d, dtype=dtype, mu=np.zeros(d), sigma=_sigma(d))
    good.sync()
    x, lp = good.current()
    # (FP32: 2 D roundings of 2^-24 times the factor's condition, sqrt(4 D / 0.1) at most: 1.4e-4)
    ref = -0.5 * np.einsum("ia,ab,ib->i", x.double().cpu().numpy(), np.linalg.inv(_sigma(d)), x.double().cpu().numpy())
    np.testing.assert_allclose(lp.double().cpu().numpy(), ref, rtol=2e-4 if dtype == torch.float32 else 1e-9)
    for col in range(d):
        for value in (-1.0, np.nan, 0.0):
            s = _sigma(d)
            # the column's pivot becomes value (its Schur complement is moved by it)
            lead = s[:col, :col]
            s[col, col] = value + (s[col, :col] @ np.linalg.solve(lead, s[:col, col]) if col else 0.0)
            if value == 0.0:
                s[col, col] -= 1e-9 * abs(s[col, col])  # (not above zero whatever the rounding)
            S = nat.Sampler(100, d, dtype=dtype, mu=np.zeros(d), sigma=s)
            with pytest.raises(nat.SmcError) as e:
                S.sync()
            assert e.value.code == nat.SMC_EINVAL, (col, value)
            S.close()
