"""The copy's source entries: one per 512 output rows up to 2^21 rows, one per
1024 above.  The host restatements of the gathering move's and the stamped
scan's rules give Algorithm 5's sources with either."""
import numpy as np
import pytest

import test_gather_sources as gather
import test_stamped_windows as stamped
from paper_1905_10252_gb300 import inputs


@pytest.mark.parametrize("rows", [512, 1024])
@pytest.mark.parametrize("n", [511, 513, 1025, 12289, 70001])
@pytest.mark.parametrize("kind", ["multinomial", "skewed", "one_hot", "ones"])
def test_either_entry_size_gives_the_sources(orc, monkeypatch, rows, n, kind):
    nc = inputs.composition(n, seed=n + 5, kind=kind)
    want = orc.redistribute(nc, np.arange(n, dtype=np.int64).reshape(n, 1)).ravel()
    monkeypatch.setattr(gather, "COPY_TILE", rows)
    monkeypatch.setattr(stamped, "RTILE", rows)
    assert np.array_equal(gather.resolve_sources(nc), want)
    for fill_all, tiles in ((1 << 17, 1024), (0, 1024), (0, 3)):
        got = stamped.stamped_sources(nc, np.random.default_rng(n), fill_all=fill_all, max_tiles=tiles)
        assert np.array_equal(got, want)
