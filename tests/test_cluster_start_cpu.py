"""Order of the cluster barrier and the first store into another block (no GPU).

A block may address another block's shared memory only once that block runs,
so the shifted-plane sweeps, which store the entering plane into the blocks
that own its shifted rows, have to meet at a cluster barrier first: an arrive
at the top of the kernel, the wait before the first store.  A sweep without it
works as long as the blocks of a cluster happen to start together, so no result
shows its absence; this test reads it off the kernels' sources.
"""

import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1701_01607_gb300", "csrc")
ARRIVE = r"\bcluster_arrive(_relaxed)?\(\)|\bcluster_barrier\(\)"
WAIT = r"\bcluster_wait(_acquire)?\(\)|\bcluster_barrier\(\)"
STORE = r"(?<!auto )\bput\("


def body(name, function):
    """The statements of a kernel body, without comments and without the lambdas
    it defines (their calls count where they are made)."""
    src = open(os.path.join(CSRC, name)).read()
    start = src.index("{", src.index(function + "(const"))
    depth, end = 0, start
    for end in range(start, len(src)):
        depth += {"{": 1, "}": -1}.get(src[end], 0)
        if depth == 0:
            break
    text = re.sub(r"//[^\n]*", "", src[start:end])
    out, pos = [], 0
    for m in re.finditer(r"auto \w+ = \[&\]\([^{]*\{", text):
        if m.start() < pos:
            continue
        out.append(text[pos:m.start()])
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
        pos = i
    return "".join(out + [text[pos:]])


@pytest.mark.parametrize("name,function,guard", [
    ("plane_sweep.cuh", "plane_sweep_body", r"if \(cl && !as\) "),
    ("plane_var.cuh", "plane_var_body", r"if \(cl\) "),
    ("ml_plane.cuh", "ml_plane_body", r"if \(cl\) "),
])
def test_cluster_meets_before_the_first_remote_store(name, function, guard):
    text = body(name, function)
    store = re.search(STORE, text).start()
    arrive = re.search(guard + "(" + ARRIVE + ")", text)
    wait = re.search(guard + "(" + WAIT + ")", text)
    assert arrive and wait and arrive.start() <= wait.start() < store


def test_counted_stores_meet_before_the_first_remote_store():
    text = body("plane_sweep.cuh", "plane_sweep_body")
    meet = re.search(r"if \(as && nz > 1\) \{\s*cluster_barrier\(\)", text)
    assert meet and meet.start() < re.search(STORE, text).start()
