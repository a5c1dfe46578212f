"""A workspace that is large enough for N particles is large enough for fewer:
a caller that allocates once for its largest N may use it for any smaller one
(the stateless calls are not told the size and rely on it)."""
import ctypes

import pytest

from paper_1905_10252_gb300 import build, native

# around every size rule of the passes: one quantise tile, the copy-count scan
# of one kernel (32 tiles of 4096), the samplers whose tiles are shared by a
# cluster of blocks (76 tiles), the cap of the covariance's blocks
EDGES = [1, 2, 127, 128, 256, 257, 512, 513, 1024, 2048, 2049, 4096, 4097, 38912, 38913, 131072, 131073, 311296,
         311297, 311500, 311700, 312000, 315392, 315393, 1 << 20, (1 << 20) + 1, 1 << 24]


@pytest.fixture(scope="module")
def lib():
    build.build()
    return native.load_library()  # (the size queries need no GPU)


def _raw(lib, n):
    out = ctypes.c_size_t()
    assert lib.smc_redistribute_ws_bytes(n, ctypes.byref(out)) == 0
    return out.value


def _sampler(lib, n, d, dtype, flags):
    cfg = native.smc_config(n=n, d=d, dtype=dtype, target=native.SMC_GAUSS, step=0.5, init_scale=2.0, flags=flags,
                            mu_dev=256, sigma_dev=512)  # (the query reads neither)
    out = ctypes.c_size_t()
    assert lib.smc_workspace_bytes(ctypes.byref(cfg), ctypes.byref(out)) == 0
    return out.value


def _check(size):
    sizes = [size(n) for n in EDGES]
    for (n0, a), (n1, b) in zip(zip(EDGES, sizes), zip(EDGES[1:], sizes[1:])):
        assert a <= b, (n0, a, n1, b)


def test_stateless_workspace_grows_with_n(lib):
    _check(lambda n: _raw(lib, n))


@pytest.mark.parametrize("d,dtype", [(1, native.SMC_F32), (8, native.SMC_F32), (32, native.SMC_F64)])
@pytest.mark.parametrize("flags", [0, native.FLAG_DEFER_REDISTRIBUTE])
def test_sampler_workspace_grows_with_n(lib, d, dtype, flags):
    _check(lambda n: _sampler(lib, n, d, dtype, flags))
