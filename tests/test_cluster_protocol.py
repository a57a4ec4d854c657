"""Distributed shared memory may be accessed only once every CTA of the cluster
is known to run, and no CTA may leave while its shared memory is still read: in
every kernel that maps a peer's shared memory a cluster barrier comes before the
first such access, and another one after the last (checked in the source, as a
violation is a race that a run need not show)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_04763_gb300", "csrc")


def _block(s, at):
    """End of the brace block that opens at or after `at`."""
    depth, i = 0, s.index("{", at)
    while True:
        depth += {"{": 1, "}": -1}.get(s[i], 0)
        i += 1
        if depth == 0:
            return i


def _kernels():
    out = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        s = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, f)).read())
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", s):
            body = s[s.index("{", m.end()):_block(s, m.end())]
            if "map_shared_rank" in body:
                out.append((m.group(1), body))
    return out


def _events(body):
    """'sync' and 'access' in the order in which the kernel's own statements reach
    them: a local function counts where it is called."""
    local = {}
    while True:
        m = re.search(r"\bauto (\w+) = \[[^\]]*\]\([^)]*\)\s*\{", body)
        if not m:
            break
        end = _block(body, m.end() - 1)
        local[m.group(1)] = body[m.end():end - 1]
        body = body[:m.start()] + body[end:].lstrip(";")
    names = "|".join(map(re.escape, local)) or "(?!)"
    token = re.compile(r"cl\.sync\(\)|map_shared_rank|\b(?:%s)\(" % names)

    def walk(text, seen):
        for t in token.findall(text):
            if t == "cl.sync()":
                yield "sync"
            elif t == "map_shared_rank":
                yield "access"
            elif t[:-1] not in seen:
                yield from walk(local[t[:-1]], seen | {t[:-1]})
    return list(walk(body, frozenset()))


def test_there_are_cluster_kernels():
    assert {"k_vcycle_cl", "k_lu_cluster"} <= {k for k, _ in _kernels()}


@pytest.mark.parametrize("name,body", _kernels(), ids=[k for k, _ in _kernels()])
def test_peers_are_accessed_between_cluster_barriers(name, body):
    ev = _events(body)
    first, last = ev.index("access"), len(ev) - 1 - ev[::-1].index("access")
    assert "sync" in ev[:first], "no cluster barrier before the first access"
    assert "sync" in ev[last + 1:], "no cluster barrier after the last access"
