"""Barriers and limits whose lack a run need not show, read from the sources.

Distributed shared memory may be accessed once every CTA of the cluster is
known to run: a kernel that maps an address of a peer CTA meets a cluster
barrier first. Votes and shuffles order no memory: lanes of a warp that change
one shared word in turn need a warp barrier between them.

A kernel's limit of dynamic shared memory belongs to the function, not to the
call: set by every call to its own size, one host thread lowers it between
another's attribute and launch. It is set once per device, to the largest size.
"""
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


def test_replicate_orders_the_takes_of_a_warp():
    """Two takes of one window may set bits of the same layer's word, and the
    lanes read those words at the window's start."""
    body = dict(kernels())["replicate_kernel"]
    window = body[body.index("for (int base = 0; base < nc; base += 32)"):]
    read = window.index("cov[lg >> 6] >>")
    loop = window.index("for (;;)")
    take = window.index("cov[lg >> 6] |=")
    assert read < window.index("__syncwarp()", read) < loop < take
    count = window.index("++count;", take)  # runs in every lane, once a take
    end = window.index("if (lane == 0)", count)
    assert window[count:end].split("}")[0].count("__syncwarp()") == 1


def test_limits_of_shared_memory_are_set_once_per_device():
    n = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"cudaFuncSetAttribute\((?!\w*\))", text):
            function = text[text.rindex("\n}", 0, m.start()):m.start()]
            assert "per_device(" in function or re.search(r"\w+_attr\(\) \{", function), (path, function[-300:])
            n += 1
    assert n >= 20
    for helper in ("ffn_attr", "router_attr", "router_lanes_attr", "place_attr"):
        calls = []
        for path in glob.glob(os.path.join(CSRC, "*.cu")):
            text = open(path).read()
            calls += [text[text.rindex("\n}", 0, m.start()):m.start()]
                      for m in re.finditer(helper + r"(<[^>]*>)?\(\)(?! \{)", text)]
        assert calls and all("per_device(" in c for c in calls), helper
