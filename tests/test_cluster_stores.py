"""Stores into another block's shared memory wait for that block (CPU: sources).

Distributed shared memory may be touched only once every block of the cluster
is known to have started, so a kernel that names ``shared::cluster`` addresses
has passed a cluster barrier before, in the order of its source.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2307_12988_gb300", "csrc")


def _kernels():
    for f in sorted(os.listdir(CSRC)):
        if f.endswith(".cu"):
            text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
            for part in re.split(r"(?=__global__)", text)[1:]:
                if "mapa.shared::cluster" in part or "st.shared::cluster" in part:
                    yield f, part


@pytest.mark.parametrize("f,body", list(_kernels()), ids=[f for f, _ in _kernels()])
def test_cluster_barrier_before_the_first_remote_store(f, body):
    first = min(body.index(w) for w in ("mapa.shared::cluster", "st.shared::cluster") if w in body)
    assert "cluster_sync();" in body[:first]
