"""The one-kernel scan of copy counts (up to 32 blocks of 4096) and the
three-pass one above it, on one workspace reused from call to call."""
import pytest
import torch

from paper_1905_10252_gb300 import inputs

pytestmark = pytest.mark.gpu

RULE = 32 * 4096


@pytest.fixture(scope="module")
def nat():
    from paper_1905_10252_gb300 import native

    native.lib()
    return native


@pytest.mark.parametrize("n", [1, 2, 511, 513, 4096, 4097, 20011, 65537, RULE - 1, RULE, RULE + 1, 300007])
def test_repeat_and_errors(nat, n):
    ws = torch.full((nat.smc_redistribute_ws_bytes(n),), 0x5A, dtype=torch.uint8, device="cuda")
    x = torch.arange(3 * n, dtype=torch.float32, device="cuda").reshape(n, 3)
    out = torch.empty_like(x)
    for kind in ("one_hot", "skewed", "ones", "multinomial"):
        nc = torch.as_tensor(inputs.composition(n, seed=n, kind=kind), device="cuda")
        ref = torch.repeat_interleave(x, nc.long(), dim=0)
        nat.smc_redistribute_raw(nc, x, out, ws)
        assert nat.smc_ws_status(ws) == nat.SMC_OK
        assert torch.equal(out, ref)
        # a wrong vector writes nothing and is reported; the next call starts afresh
        out.fill_(-1.0)
        bad = nc.clone()
        bad[n // 2] = -1 if kind == "ones" else bad[n // 2] + 1
        nat.smc_redistribute_raw(bad, x, out, ws)
        assert nat.smc_ws_status(ws) == nat.SMC_EINVAL and bool((out == -1.0).all())
        nat.smc_redistribute_raw(bad, x, out, ws)
        nat.smc_redistribute_raw(nc, x, out, ws)
        assert nat.smc_ws_status(ws) == nat.SMC_OK and torch.equal(out, ref)
        if n <= 1 << 20:
            out.fill_(-1.0)
            status = torch.full((1,), 7, dtype=torch.int32, device="cuda")
            nat.smc_redistribute_raw_noalloc(nc, x, out, status)
            assert int(status) == nat.SMC_OK and torch.equal(out, ref)


@pytest.mark.parametrize("n", [3000, RULE - 5, RULE + 5])
def test_sampler_redistribute_between_iterations(nat, n):
    """The sampler's run-start array stays clean for the iterations that follow
    an explicit redistribution."""
    mu, sigma = inputs.gaussian_target(5, seed=5)
    a, b = (nat.Sampler(n, 5, seed=3, mu=mu, sigma=sigma, resample_mode=nat.RESAMPLE_ALWAYS) for _ in range(2))
    a.step(1)
    b.move()
    b.reweight()
    nc, _ = b.resample()
    b.redistribute(nc)
    for s in (a, b):
        s.step(3)
        s.sync()
    for u, v in zip(a.current(), b.current()):
        assert torch.equal(u, v)
