"""A run's iterations in one call or in several: plain launches, graphs of one
and of eight give the same bits, whichever of them a call's length selects
(the rules' edges: 8 and 24 iterations run, 8 and 16 left in the call)."""
import pytest
import torch

from paper_1905_10252_gb300 import inputs

pytestmark = pytest.mark.gpu

TOTAL = 58
SPLITS = [[58], [20, 20, 18], [8, 15, 16, 19], [23, 8, 27], [24, 7, 8, 1, 9, 9], [7, 16, 17, 1, 17], [1] * 58]


def _run(dtype, mode, splits, cov):
    from paper_1905_10252_gb300 import native as nat

    mu, sigma = inputs.gaussian_target(3, seed=2)
    s = nat.Sampler(5003, 3, seed=4, mu=mu, sigma=sigma, dtype=dtype, resample_mode=mode)
    for k in splits:
        out = s.step(k, cov=cov)
    s.sync()
    res = [*s.current(), s.logw, out["mean"]] + ([out["cov"]] if cov else [])
    return [t.clone() for t in res]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("cov", [False, True])
def test_splits_agree(dtype, mode, cov):
    ref = _run(dtype, mode, SPLITS[-1], cov)
    for splits in SPLITS[:-1]:
        assert sum(splits) == TOTAL
        for u, v in zip(ref, _run(dtype, mode, splits, cov)):
            assert torch.equal(u, v), splits
