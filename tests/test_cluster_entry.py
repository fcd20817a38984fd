"""Kernels that write the shared memory of other CTAs of their cluster (CPU: the source is read, nothing is launched).

A CTA's distributed shared memory may be accessed only once that CTA has started, so a cluster-wide barrier has to
come before the first remote access of a kernel, and another one after the last."""
import os
import re

import pytest

import paper_2609_21633_gb300 as tn

CSRC = os.path.join(os.path.dirname(os.path.abspath(tn.__file__)), "csrc")


def _kernels():
    """(name, body without comments) of every __global__ function that maps another CTA's shared memory."""
    out = []
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, f)).read(), flags=re.S)
        for m in re.finditer(r"__global__\s+void[^{;]*?(k_\w+)\s*\([^{;]*\)\s*\{", src):
            depth, e = 1, m.end()
            while depth:
                depth += {"{": 1, "}": -1}.get(src[e], 0)
                e += 1
            body = src[m.end():e - 1]
            if "map_shared_rank" in body:
                out.append((m.group(1), body))
    return out


def test_some_kernel_is_found():
    assert "k_cg_cluster" in [k for k, _ in _kernels()]


@pytest.mark.parametrize("name,body", _kernels(), ids=lambda v: v if len(v) < 40 else "")
def test_cluster_barrier_before_the_first_remote_access_and_after_the_last(name, body):
    # the kernel's lambdas, and those of them through which remote memory is reached
    lambdas = re.findall(r"auto (\w+) = \[&\](.*?)\n  \};", body, flags=re.S)
    remote = {n for n, b in lambdas if "map_shared_rank" in b}
    while True:
        more = {n for n, b in lambdas if n not in remote and any(re.search(r"\b%s\(" % r, b) for r in remote)}
        if not more:
            break
        remote |= more
    straight = re.sub(r"auto (\w+) = \[&\](.*?)\n  \};", "", body, flags=re.S)
    uses = [m.start() for r in remote | {"map_shared_rank"} for m in re.finditer(r"\b%s\(" % r, straight)]
    syncs = [m.start() for m in re.finditer(r"\bcl\.sync\(\)", straight)]
    assert uses and syncs
    assert min(syncs) < min(uses), "%s: remote shared memory is reached before the cluster has met" % name
    assert max(syncs) > max(uses), "%s: a CTA may leave while its shared memory is still written" % name
