"""A CTA may touch another CTA's shared memory only once that CTA is known to have started,
which a completed cluster barrier says: in every kernel that maps a peer's shared memory,
cl.sync() or cl.barrier_wait() stands before the first access in program order (the body of
a lambda counts where it is called).  Read from the sources: a CTA that is late by chance
cannot be staged on a GPU.
"""
import glob
import os
import re

import pytest

from conftest import ROOT


def _block(text, at):
    """The braced block that opens at or after `at`: (start, end) of its inside."""
    start = text.index("{", at)
    depth = 0
    for k in range(start, len(text)):
        depth += {"{": 1, "}": -1}.get(text[k], 0)
        if depth == 0:
            return start + 1, k
    raise ValueError("unbalanced braces")


def _kernels():
    out = []
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_2404_06260_gb300/csrc/*.cu"))):
        text = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)
        for m in re.finditer(r"__global__\s+void", text):
            name = re.search(r"(k_\w+)\s*\(", text[m.end():]).group(1)
            a, b = _block(text, text.index(name, m.end()))
            if "map_shared_rank" in text[a:b]:
                out.append(pytest.param(text[a:b], id=name))
    return out


def _flat(body):
    """The body with every lambda's block moved to the places that call it."""
    while True:
        m = re.search(r"auto\s+(\w+)\s*=\s*\[[^\]]*\]\s*\((?:[^()]|\([^()]*\))*\)\s*(?=\{)", body)
        if not m:
            return body
        a, b = _block(body, m.end())
        inner, rest = body[a:b], body[:m.start()] + body[b + 1:]
        body = re.sub(r"\b%s\(" % m.group(1), lambda _: "{" + inner + "}(", rest)


@pytest.mark.parametrize("body", _kernels())
def test_cluster_barrier_before_the_first_remote_access(body):
    body = _flat(body)
    first = body.index("map_shared_rank")
    waits = [body.find(w) for w in ("cl.sync()", "cl.barrier_wait()") if w in body]
    assert waits and min(waits) < first
    # a wait needs its arrival, and nothing leaves the kernel between the two
    if "cl.barrier_wait()" in body:
        arrive = body.index("cl.barrier_arrive()")
        assert arrive < body.index("cl.barrier_wait()")
        assert "return" not in body[arrive:body.index("cl.barrier_wait()")]


def test_the_cluster_kernels_are_found():
    assert {p.id for p in _kernels()} >= {"k_rcg_cluster", "k_sym_eig_blocks", "k_cg_resident",
                                          "k_cg_coarse_tc"}
