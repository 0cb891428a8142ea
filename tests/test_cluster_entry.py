"""Cluster kernels meet before they touch each other's shared memory.

CUDA leaves an access to the shared memory of a CTA that has not started yet
undefined, and nothing but a cluster barrier says that it has.  The order is
read off the kernel sources: in every device function that maps a remote shared
address, a cluster barrier comes first, lambdas counted where they are called.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2312_02999_gb300", "csrc")
REMOTE = "map_shared_rank"
BARRIERS = (r"\bcl\.sync\s*\(", r"\bbarrier_wait\s*\(")


def _block(text, start):
    """The brace block that opens at or after start: (first, past the end)."""
    i = text.index("{", start)
    depth = 0
    for k in range(i, len(text)):
        depth += (text[k] == "{") - (text[k] == "}")
        if depth == 0:
            return i, k + 1
    raise ValueError("unbalanced braces")


def _events(body, lambdas):
    """Barriers and remote accesses of a body in the order they run."""
    found = [(m.start(), "barrier") for p in BARRIERS for m in re.finditer(p, body)]
    found += [(m.start(), "remote") for m in re.finditer(REMOTE, body)]
    for name, inner in lambdas.items():
        for m in re.finditer(r"\b%s\s*\(" % name, body):
            found += [(m.start(), e) for e in inner]
    return [e for _, e in sorted(found, key=lambda f: f[0])]


def _functions():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"^__(?:device|global)__[^;{]*?(\w+)\s*\([^;{]*\)\s*\{", text, re.M):
            a, z = _block(text, m.end() - 1)
            if REMOTE in text[a:z]:
                yield os.path.basename(path), m.group(1), text[a:z]


def _first_event(body):
    lambdas = {}
    while True:
        m = re.search(r"\bauto\s+(\w+)\s*=\s*\[&\]", body)
        if not m:
            break
        a, z = _block(body, m.end())
        lambdas[m.group(1)] = _events(body[a:z], lambdas)
        body = body[:m.start()] + body[z:]
    events = _events(body, lambdas)
    return events[0] if events else None


@pytest.mark.parametrize("where", [(f, n) for f, n, _ in _functions()])
def test_barrier_before_remote_shared_memory(where):
    bodies = {(f, n): b for f, n, b in _functions()}
    assert _first_event(bodies[where]) == "barrier", where


def test_every_user_is_looked_at():
    names = {n for _, n, _ in _functions()}
    assert {"k_small_solve_body", "k_clus_v_body"} <= names
