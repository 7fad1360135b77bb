"""The order of a cluster kernel's first accesses to its peer's shared memory,
checked on the source: a missing barrier there is a race that shows only when
the peer CTA starts late, so no run can be relied on to fail for it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_10302_gb300", "csrc")
SYNC, MAP = "this_cluster().sync()", "map_shared_rank("


def _functions(src):
    """Name -> body of every function defined at file scope."""
    out = {}
    for m in re.finditer(r"\b(\w+)\((?:[^(){};]|\([^()]*\))*\)\s*\{", src):
        if m.group(1) in ("if", "for", "while", "switch"):
            continue
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        out.setdefault(m.group(1), src[m.end():i - 1])
    return out


def _cluster_ops(name, funcs, seen=()):
    """The cluster barriers and peer mappings of a function and of what it
    calls, in the order of the text."""
    ops = []
    for m in re.finditer(r"this_cluster\(\)\.sync\(\)|map_shared_rank\(|\b(\w+)(?:<[^;(){}]*>)?\(", funcs[name]):
        if m.group(0) in (SYNC, MAP):
            ops.append(m.group(0))
        elif m.group(1) in funcs and m.group(1) not in seen and m.group(1) != name:
            ops += _cluster_ops(m.group(1), funcs, (*seen, name))
    return ops


@pytest.mark.parametrize("path,kernel", [("apt.cu", "apt_kernel"), ("graph.cu", "gapt_kernel")])
def test_a_cluster_barrier_precedes_the_first_access_to_the_peer(path, kernel):
    src = open(os.path.join(CSRC, path)).read()
    src = re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)
    ops = _cluster_ops(kernel, _functions(src))
    assert ops.count(MAP) >= 2 and ops.count(SYNC) >= 2   # the walk found them
    assert ops[0] == SYNC, ops
    assert ops[-1] == SYNC, ops                           # nor does a CTA leave while its peer may still reach it
