"""The cluster reduce and the 512-item scan of samplers of few tiles against
the one-block-per-tile passes (which a batch uses at every size): the same
bits, at the edges of the tiles, their eighths and the rule between them."""
import pytest
import torch

from paper_1905_10252_gb300 import inputs

pytestmark = pytest.mark.gpu

TILE, RULE = 4096, 76


@pytest.fixture(scope="module")
def nat():
    from paper_1905_10252_gb300 import native

    native.lib()
    return native


def _sampler(nat, n, d, mode, seed=9):
    mu, sigma = inputs.gaussian_target(d, seed=d)
    return nat.Sampler(n, d, seed=seed, mu=mu, sigma=sigma, resample_mode=mode)


@pytest.mark.parametrize("n,d", [(1, 2), (511, 3), (513, 8), (4095, 32), (4097, 31), (4608, 17), (2 * TILE + 1, 4),
                                 (20011, 32), (5 * TILE - 1, 9), (RULE * TILE, 7), (RULE * TILE + 1, 7),
                                 (RULE * TILE - 511, 24), (100 * TILE + 77, 32), (90 * TILE + 5, 8)])
@pytest.mark.parametrize("mode", [0, 1, 2])
def test_solo_and_batched_passes_agree(nat, n, d, mode):
    a, b = _sampler(nat, n, d, mode), _sampler(nat, n, d, mode)
    oa = a.step(3, trace=True, fhat=True)
    batch = nat.Batch([b])
    ob = batch.step(3, trace=True, fhat=True)
    batch.sync()
    a.sync()
    for u, v in zip(a.current(), b.current()):
        assert torch.equal(u, v)
    assert torch.equal(a.logw, b.logw)
    assert torch.equal(oa["mean"], ob["mean"][0]) and torch.equal(oa["fhat"], ob["fhat"][0])
    assert torch.equal(oa["trace"].view(torch.int64), ob["trace"][0].view(torch.int64))
    # copy counts of W as the batched reduce left it (no prefixes inside a tile) and as the cluster did
    na, nb = a.resample()[0], b.resample()[0]
    a.sync()
    b.sync()
    if mode == 2:
        assert torch.equal(na, nb) and int(na.sum()) == n


@pytest.mark.parametrize("n,d", [(700, 5), (5000, 16), (9001, 32), (30000, 2), (RULE * TILE + 9, 4)])
def test_fp64_estimate_against_sums(nat, n, d):
    """FP64 samplers (every route of the cluster pass's columns): eq. (7)
    within the rounding of N terms."""
    mu, sigma = inputs.gaussian_target(d, seed=d)
    s = nat.Sampler(n, d, dtype=torch.float64, seed=4, mu=mu, sigma=sigma)
    s.move()
    s.reweight()
    mean, _ = s.estimate()
    x, lw = s.current()[0], s.logw
    w = torch.exp(lw - lw.max())
    ref, mag = (w @ x) / w.sum(), (w @ x.abs()) / w.sum()
    assert bool(((mean - ref).abs() <= 2.0**-44 * mag + n * 7.8e-20 * x.abs().max()).all())
