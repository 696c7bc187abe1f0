"""Cluster kernels: a block may touch another's shared memory only after a cluster
barrier has shown that every block of the cluster runs (host-only, by reading the
source: the barrier stands before the item loop, whose first turn stores there)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2202_07017_gb300", "csrc")


def _cluster_kernels():
    """(name, body) of every kernel with __cluster_dims__."""
    found = []
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"__cluster_dims__\([^)]*\).*?(\w+)\(const", text, re.S):
            body = text[text.index("{", m.end()):]
            found.append((m.group(1), body[:body.index("\n}\n")]))
    return found


def test_cluster_kernels_are_found():
    assert sorted(name for name, _ in _cluster_kernels()) == ["kbatch_cl", "kbatch_wide"]


@pytest.mark.parametrize("kernel", ["kbatch_cl", "kbatch_wide"])
def test_a_cluster_barrier_before_the_first_remote_access(kernel):
    body = dict(_cluster_kernels())[kernel]
    barrier, loop = body.index("cluster.sync()"), body.index("while (true)")
    assert barrier < loop
    # and no address of another block is used up to there
    assert not re.search(r"\*\s*cluster\.map_shared_rank|\*partner", body[:barrier])
