"""smc_step inside a caller's own stream capture: whichever of its graphs the
sampler has built before, the call is captured and its replays continue the
run with the bits of plain calls."""
import pytest
import torch

from paper_1905_10252_gb300 import inputs

pytestmark = pytest.mark.gpu


def _sampler(dtype, n=5003, d=3):
    from paper_1905_10252_gb300 import native as nat

    mu, sigma = inputs.gaussian_target(d, seed=2)
    return nat.Sampler(n, d, seed=4, mu=mu, sigma=sigma, dtype=dtype)


def _state(s):
    s.sync()
    return [t.clone() for t in (*s.current(), s.logw)]


# iterations before the capture: none of the graphs, that of eight, both
@pytest.mark.parametrize("before", [[3], [8, 16], [24, 24, 1]])
@pytest.mark.parametrize("cov", [False, True])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_captured_step_continues_the_run(dtype, cov, before):
    k, replays = 11, 3
    a, b = _sampler(dtype), _sampler(dtype)
    for n in before:
        a.step(n)
        b.step(n)
    a.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=a.stream):
        out = a.step(k, cov=cov)
    for _ in range(replays):
        with torch.cuda.stream(a.stream):
            g.replay()
        ref = b.step(k, cov=cov)
    for u, v in zip(_state(a), _state(b)):
        assert torch.equal(u, v)
    assert torch.equal(out["mean"], ref["mean"])
    if cov:
        assert torch.equal(out["cov"], ref["cov"])
    # and the sampler goes on outside the capture
    a.step(20)
    b.step(20)
    for u, v in zip(_state(a), _state(b)):
        assert torch.equal(u, v)
