"""Distributed shared memory may be accessed once every CTA of the cluster is
known to run: a kernel that maps an address of a peer CTA meets a cluster
barrier first (read from the sources, since a run need not show its lack)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_17154_gb300", "csrc")


def kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__[^;{]*?(\w+)\(\s*(?:const|int|uint)", text):
            depth, start = 0, text.index("{", m.end())
            for i in range(start, len(text)):
                depth += {"{": 1, "}": -1}.get(text[i], 0)
                if depth == 0:
                    break
            yield m.group(1), text[start:i]


PEERS = [(n, b) for n, b in kernels() if "mapa_shared(" in b]


def test_kernels_with_peers_are_found():
    assert {n for n, _ in PEERS} == {"router_select_kernel", "router_lanes_kernel", "ffn_gemm_kernel",
                                     "sim_logits_kernel"}


@pytest.mark.parametrize("name,body", PEERS, ids=[n for n, _ in PEERS])
def test_cluster_barrier_before_the_first_access_to_a_peer(name, body):
    first = body.index("mapa_shared(")
    assert 0 <= body.find("cluster_sync()") < first, name
