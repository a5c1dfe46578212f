"""The tensor-core logistic likelihood at the edges of its tiles: an odd number
of 128-particle tiles (the last pass holds one), CTAs with one and with two
tiles, one and several image tiles of 256 rows, and the flush after eight."""
import numpy as np
import pytest
import torch

from paper_1905_10252_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_1905_10252_gb300 import native

    native.lib()
    return native


@pytest.mark.parametrize("n,m,d", [(1, 1, 1), (128, 128, 16), (129, 129, 32), (257, 256, 17), (384, 257, 4),
                                   (152 * 128, 300, 9), (152 * 128 + 1, 513, 31), (303 * 128, 2048, 5),
                                   (305 * 128 - 5, 2304, 32), (457 * 128 + 3, 2305, 12)])
def test_logpi_at_tile_edges(nat, n, m, d):
    X, y, _ = inputs.logistic_data(m, d, seed=n + m)
    S = nat.Sampler(n, d, seed=11, target="logistic", X=X, y=y, prior_var=4.0, step=0.2,
                    resample_mode=nat.RESAMPLE_NEVER)
    S.move()
    S.reweight()
    S.sync()
    x, lp = S.current()
    Xd, yd = torch.from_numpy(X).cuda().double(), torch.from_numpy(y).cuda().double()
    worst = 0.0
    for a in range(0, n, 8192):
        b = x[a:a + 8192].double()
        z = b @ Xd.T
        ref = z @ yd - torch.logaddexp(z, torch.zeros_like(z)).sum(1) - (b * b).sum(1) / 8.0
        # 2^-16 of every product (the split), the epilogue's approximations
        # per row, half an ulp of the FP32 result
        bound = 2.0**-16 * (b.abs() @ Xd.abs().T).sum(1) + 2e-6 * m + 2.0**-24 * ref.abs()
        worst = max(worst, float(((lp[a:a + 8192].double() - ref).abs() / bound).max()))
    assert worst <= 1.0
