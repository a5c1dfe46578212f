"""The FP64 target's division by a known divisor: the same bits as IEEE
division over the exponent range, where it takes its short form and where it
divides as usual (log pi = -1/2 ((x - mu) / L)^2 for D = 1)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [700, 20000])
@pytest.mark.parametrize("init,var", [(2.0, 1.7), (1e-250, 1.0), (1e-120, 3e-300), (1e120, 7e250), (1e5, 1e-300),
                                      (1e-3, 2e300), (1.3e140, 5e-3), (3e-200, 1.1e-200)])
def test_known_divisor(n, init, var):
    from paper_1905_10252_gb300 import native as nat

    s = nat.Sampler(n, 1, dtype=torch.float64, seed=int(abs(np.log10(var))) + n, mu=[0.0], sigma=[[var]], step=0.0,
                    init_scale=init)
    x, lp = (t.cpu().numpy().ravel() for t in s.current())
    with np.errstate(all="ignore"):
        z = x / np.sqrt(np.float64(var))
        ref = -0.5 * (z * z)
    assert np.array_equal(lp, ref)
