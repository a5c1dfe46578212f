"""smc_step's one-launch iterations of small FP64 samplers, at the sizes that
take them: D <= 2 up to N = 512 and D = 3 up to 256, unless every iteration
resamples.  Which path a sampler takes is shown by the test hook that stalls
the launch's grid barrier; the results must equal, bit for bit, the same
iterations launched stage by stage, and the oracle's run."""
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


def host(t):
    return t.detach().cpu().numpy()


def _make(nat, n, d, seed, mode=0, **kw):
    if kw.pop("student", False):
        return nat.Sampler(n, 1, dtype=torch.float64, seed=seed, target="student_t", mu=1.5, nu=5.0, step=0.5,
                           init_scale=2.0, resample_mode=mode, **kw)
    mu, sig = inputs.gaussian_target(d, seed=40 + d)
    return nat.Sampler(n, d, dtype=torch.float64, seed=seed, mu=mu, sigma=sig, step=0.5, init_scale=2.0,
                       resample_mode=mode, **kw)


def _state(S):
    S.sync()
    return [t.clone() for t in (*S.current(), S.logw)]


@pytest.mark.parametrize("n,d,mode,fused", [
    (1, 1, 0, True), (512, 1, 0, True), (513, 1, 0, False), (512, 2, 0, True), (513, 2, 0, False),
    (256, 3, 0, True), (257, 3, 0, False), (512, 2, 2, True), (256, 4, 0, False), (64, 5, 0, False),
    (64, 32, 0, False), (64, 1, 1, False), (256, 2, 1, False)])
def test_which_samplers_take_the_one_launch(nat, n, d, mode, fused):
    S = _make(nat, n, d, 1, mode, flags=nat.FLAG_TEST_STALL_BARRIER)
    S.step(1 if n == 1 else 2)
    if fused:
        with pytest.raises(nat.SmcError) as e:
            S.sync()
        assert e.value.code == nat.SMC_ETIMEOUT
    else:
        S.sync()
    S.close()


SIZES = [(1, 1), (2, 2), (31, 3), (32, 1), (33, 2), (255, 3), (256, 3), (255, 1), (256, 2), (257, 1), (300, 2),
         (511, 1), (512, 2)]


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("n,d", SIZES)
def test_equals_stage_launches(nat, n, d, mode):
    K = 9
    a, b, c = (_make(nat, n, d, 11, mode) for _ in range(3))
    ra = a.step(K, cov=True, trace=True, fhat=True)
    for _ in range(K):
        b.step_profile()
    for u, v in zip(_state(a), _state(b)):
        assert torch.equal(u, v)
    sa, sb = a.stats(), b.stats()
    for key in ("lse", "logc", "ess", "max_logw", "resampled", "t", "survivors"):
        assert sa[key] == sb[key] or (np.isnan(sa[key]) and np.isnan(sb[key])), key
    # in two calls, and the covariance from the separate calls' last iteration
    c.step(5)
    c.step(K - 6)
    c.move()
    c.reweight()
    mean, cov = c.estimate(cov=True)
    c.sync()
    assert torch.equal(ra["mean"], mean) and torch.equal(ra["cov"], cov)
    for S in (a, b, c):
        S.close()


@pytest.mark.parametrize("n", [7, 256, 300, 512])
def test_student_t_equals_stage_launches(nat, n):
    a, b = _make(nat, n, 1, 5, student=True), _make(nat, n, 1, 5, student=True)
    a.step(12)
    for _ in range(12):
        b.step_profile()
    for u, v in zip(_state(a), _state(b)):
        assert torch.equal(u, v)


@pytest.mark.parametrize("n,d,seed", [(512, 2, 3), (333, 1, 5), (256, 3, 7), (100, 3, 2)])
def test_against_oracle(nat, orc, n, d, seed):
    K = 12
    mu, sig = inputs.gaussian_target(d, seed=40 + d)
    ref = orc.run(orc.Target.gauss(mu, sig), n, seed, K, init_scale=2.0, step=0.5, ncopies_trace=True)
    S = _make(nat, n, d, seed)
    out = S.step(K, cov=True, trace=True, fhat=True)
    S.sync()
    x, lp = S.current()
    assert np.array_equal(host(x), ref["x"])
    assert np.array_equal(host(lp), ref["logpi"])
    assert np.array_equal(host(S.logw), ref["logw"])
    tr = nat.trace_dicts(out["trace"])
    for k in range(K):
        assert tr[k]["resampled"] == int(ref["trace"][k, 4]), k
        assert abs(tr[k]["lse"] - ref["trace"][k, 0]) <= 1e-10, k
        assert tr[k]["max_logw"] == ref["trace"][k, 3], k
        assert tr[k]["survivors"] == int(ref["trace"][k, 5]), k
    np.testing.assert_allclose(host(out["mean"]), ref["means"][-1], rtol=0, atol=1e-11)
    np.testing.assert_allclose(host(out["cov"]), ref["cov"], rtol=0, atol=1e-9)
    np.testing.assert_allclose(host(out["fhat"]), ref["fhat"], rtol=0, atol=1e-10)
    S.close()
