"""Copies on both sides of 2^21 rows, where the rows per source entry (and per
copy block) go from 512 to 1024: stateless calls on one workspace, a sampler's
own and deferred copies, and a member of a batch."""
import numpy as np
import pytest
import torch

from paper_1905_10252_gb300 import inputs

pytestmark = pytest.mark.gpu

RULE = 1 << 21


@pytest.fixture(scope="module")
def nat():
    from paper_1905_10252_gb300 import build, native

    build.build()
    native.lib()
    return native


def _counts(n, kind):
    if kind != "few":
        return inputs.composition(n, seed=n % 1000, kind=kind)
    # about a hundred survivors close together: windows of 2^20 rows with few run starts
    rng = np.random.default_rng(n)
    c = np.zeros(n, np.int32)
    at = np.unique(np.concatenate([rng.integers(0, 8192, 60), rng.integers(n - 9000, n, 60)]))
    c[at] = rng.multinomial(n, rng.dirichlet(np.full(len(at), 0.3)))
    return c


def test_stateless_copies(nat):
    sizes = [RULE + 1025, RULE - 1, RULE, RULE + 1, RULE + 513, 3 * RULE + 7, RULE + 3]
    ws = torch.full((nat.smc_redistribute_ws_bytes(max(sizes)),), 0x5A, dtype=torch.uint8, device="cuda")
    for n in sizes:
        x = torch.arange(n, dtype=torch.int32, device="cuda").reshape(n, 1).float()
        out = torch.empty_like(x)
        for kind in ("few", "one_hot", "skewed", "ones", "multinomial"):
            nc = torch.as_tensor(_counts(n, kind), device="cuda")
            ref = torch.repeat_interleave(x, nc.long(), dim=0)
            nat.smc_redistribute_raw(nc, x, out, ws)
            assert nat.smc_ws_status(ws) == nat.SMC_OK
            assert torch.equal(out, ref), (n, kind)


@pytest.mark.parametrize("n", [RULE, RULE + 1, RULE + 1537])
def test_sampler_copies(nat, n):
    mu, sigma = inputs.gaussian_target(2, seed=5)

    def make(flags=0, mode=nat.RESAMPLE_ALWAYS):
        return nat.Sampler(n, 2, seed=3, mu=mu, sigma=sigma, resample_mode=mode, flags=flags)

    a, b, c = make(), make(nat.FLAG_DEFER_REDISTRIBUTE), make()
    m = make()
    small = nat.Sampler(3000, 2, seed=3, mu=mu, sigma=sigma, resample_mode=nat.RESAMPLE_ALWAYS)
    batch = nat.Batch([m, small])
    a.step(1)
    b.step(1)
    batch.step(1)
    c.move()
    c.reweight()
    nc, _ = c.resample()
    ref = torch.repeat_interleave(c.current()[0], nc.long(), dim=0)
    c.redistribute(nc)
    assert torch.equal(c.current()[0], ref)
    for k in (0, 3):
        if k:
            a.step(k)
            b.step(k)
            c.step(k)
            batch.step(k)
        batch.sync()
        a.sync()
        for s in (b, c, m):
            s.sync()
            for u, v in zip((*a.current(), a.logw), (*s.current(), s.logw)):
                assert torch.equal(u, v)
