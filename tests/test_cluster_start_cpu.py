"""A CTA of a thread-block cluster may write a peer's shared memory only once that peer is known to
run, which the first cluster barrier of the kernel is what guarantees, and a CTA may leave only when
no peer can write to it any more.  No run shows a missing barrier reliably, so the kernels' sources
are read: in every kernel that addresses distributed shared memory, itself or through the routine it
calls for an instance, a cluster barrier comes first, and one stands between the last such access
and each way out."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_12344_gb300", "csrc")
SYNC = "cl.sync()"
REMOTE = re.compile(r"map_shared_rank|\bsolve_one<false|\bdelta_group\(")


def _kernels():
    """(file, body) of every kernel that uses distributed shared memory, comments taken out."""
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith(".cu"):
            continue
        with open(os.path.join(CSRC, name)) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__[^{;]*\{", text):
            depth, end = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
            body = text[m.end():end]
            if "this_cluster()" in body and REMOTE.search(body):
                yield pytest.param(body, id=f"{name}:{re.search(r'(\w+)\s*\([^()]*\)\s*{$', m.group(0)).group(1)}")


KERNELS = list(_kernels())


def test_the_cluster_kernels_are_found():
    assert {p.id.split(":")[0] for p in KERNELS} >= {"dense_group.cu", "dense_mixed.cu"}


@pytest.mark.parametrize("body", KERNELS)
def test_a_cluster_barrier_precedes_the_first_remote_access(body):
    assert SYNC in body[:REMOTE.search(body).start()]


@pytest.mark.parametrize("body", KERNELS)
def test_a_cluster_barrier_precedes_every_exit(body):
    exits = [m.start() for m in re.finditer(r"\breturn\b", body)] + [len(body)]
    for at in exits:
        before = [m.end() for m in REMOTE.finditer(body[:at])]
        assert not before or SYNC in body[before[-1]:at]
