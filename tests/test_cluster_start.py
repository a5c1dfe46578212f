"""Shared memory of another block of a cluster may only be accessed once that
block has started, and must not be left before the accesses are done: a kernel
launched over clusters arrives at a cluster barrier on entry, waits for it
before its first remote store, and ends the stores with a second barrier.  A
missing wait shows on no result that can be relied on, so the order is read
from the source."""
import re
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_1905_10252_gb300" / "csrc"


def _cluster_kernels():
    """(name, body) of every kernel compiled for clusters."""
    out = []
    for src in sorted(CSRC.glob("*.cu")):
        text = re.sub(r"//[^\n]*", "", src.read_text())
        for m in re.finditer(r"__cluster_dims__\([^)]*\)\s+(\w+)\([^)]*\)\s*\{", text):
            depth, at = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[at], 0)
                at += 1
            out.append((m.group(1), text[m.end():at]))
    return out


KERNELS = _cluster_kernels()


def test_there_are_cluster_kernels():
    assert [name for name, _ in KERNELS] == ["k_quant_reduce_cluster"]


@pytest.mark.parametrize("name,body", KERNELS, ids=[k for k, _ in KERNELS])
def test_remote_stores_lie_between_two_cluster_barriers(name, body):
    stores = [m.start() for m in re.finditer(r"\bst_rank0\(", body)]
    arrive = [m.start() for m in re.finditer(r"\bcluster_arrive_started\(\)", body)]
    wait = [m.start() for m in re.finditer(r"\bcluster_wait_started\(\)", body)]
    end = [m.start() for m in re.finditer(r"\bcluster_sync\(\)", body)]
    assert stores and len(arrive) == len(wait) == len(end) == 1, name
    assert arrive[0] < wait[0] < min(stores) and max(stores) < end[0], name
    # every thread passes all three: no block of the kernel is left before the
    # last, and none of them lies inside a branch or a loop
    assert "return" not in body[: end[0]], name
    for at in (arrive[0], wait[0], end[0]):
        assert body[:at].count("{") == body[:at].count("}"), (name, at)
        assert body[:at].rstrip()[-1:] in ("", ";", "}"), (name, at)
