"""The tensor-core likelihood at values without a finite log-target: a NaN or
infinite coordinate is reported."""
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
