"""Batches and slots whose members are all narrow, all wide, of the width that
has a kernel of its own, or mixed take different kernels; every member's
results are those of its own steps."""
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


def _make(nat, n, d, mode=0):
    mu, sigma = inputs.gaussian_target(d, seed=40 + d)
    return nat.Sampler(n, d, seed=n + d, mu=mu, sigma=sigma, resample_mode=mode)


def _equal(s, k, nat, mode=0):
    ref = _make(nat, s.n, s.d, mode)
    ref.step(k)
    for t in (s, ref):
        t.sync()
    for u, v in zip((*s.current(), s.logw), (*ref.current(), ref.logw)):
        assert torch.equal(u, v), (s.n, s.d)
    a, b = s.stats(), ref.stats()
    assert all(a[key] == b[key] for key in a), (s.n, s.d)
    ref.close()


WIDTHS = [[8], [8, 8, 8], [1, 3, 7], [16], [2, 8, 16], [17], [32, 32], [9, 8, 32], [16, 17, 8, 1, 31, 32]]


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("widths", WIDTHS, ids=str)
def test_batch_members_equal_their_own_steps(nat, widths, mode):
    sizes = [5003, 1024, 300, 40961, 1, 8192]
    members = [_make(nat, n, d, mode) for n, d in zip(sizes, widths)]
    batch = nat.Batch(members)
    batch.step(4)
    batch.sync()
    for m in members:
        _equal(m, 4, nat, mode)
    batch.close()


def test_slots_change_widths_between_steps(nat):
    caps = [6000, 5000, 70000]
    slots = nat.Slots(caps)
    a, b, c = _make(nat, 5003, 8), _make(nat, 4097, 16), _make(nat, 65537, 3)
    for i, s in enumerate((a, b, c)):
        slots.attach(i, s)
    slots.step([3, 3, 3])  # narrow
    slots.sync()
    slots.detach(1)
    w = _make(nat, 4999, 32)
    slots.attach(1, w)
    slots.step([2, 2, 2])  # mixed
    slots.sync()
    slots.detach(1)
    slots.step([2, 0, 2])  # narrow again
    slots.sync()
    slots.detach(0)
    slots.detach(2)
    v = _make(nat, 60001, 17)
    slots.attach(2, v)
    slots.step([0, 0, 3])  # wide alone
    slots.sync()
    for s, k in ((a, 7), (b, 3), (c, 7), (w, 2), (v, 3)):
        _equal(s, k, nat)
    slots.close()
