"""Distributed shared memory without a GPU, by the source: another CTA's
shared memory may be accessed only once that CTA runs, so in every kernel that
maps it, all threads of all CTAs must have met at a cluster barrier before the
first statement that may store to it or load from it."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1409_2081_gb300", "csrc")
REMOTE = r"recv_of|recvd_of|map_shared_rank|cl_reduce|sums64\(\)|bcl_sums"
BARRIER = r"\bcl\.sync\(\)|\bbcl_started\(|\bcl\.barrier_wait\("


def block(src, at):
    """From the brace at or after `at` to the one that closes it."""
    i = src.index("{", at)
    depth = 0
    for j in range(i, len(src)):
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        if depth == 0:
            return i, j + 1
    raise ValueError("unbalanced braces")


def kernels():
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
        for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", src):
            i, j = block(src, m.end())
            body = src[i:j]
            if "map_shared_rank" in body:
                yield m.group(1), body


def statements(body):
    """The kernel's own statements in order: without the bodies of its lambdas
    (they run where they are called) and the address maps themselves."""
    while True:
        m = re.search(r"=\s*\[[&=]?\]\s*\([^)]*\)\s*(?=\{)", body)
        if not m:
            break
        _, j = block(body, m.end())
        body = body[:m.start()] + "= 0" + body[j:]
    body = re.sub(r"st\.recvd?_of\[[^]]*\]\s*=\s*cl\.map_shared_rank\([^;]*;", "", body)
    return re.split(r"[;{}]", body)


KERNELS = dict(kernels())


def test_kernels_found():
    assert {"k_band_pipe", "k_band_cl", "k_cg_zone_cl"} <= set(KERNELS)


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_barrier_before_the_first_access(name):
    met = False
    for s in statements(KERNELS[name]):
        if re.search(REMOTE, s):
            assert met, s.strip()
            return
        met = met or re.search(BARRIER, s) is not None
    raise AssertionError("no access found")


@pytest.mark.parametrize("name", ["k_band_pipe", "k_band_cl"])
def test_split_barrier_is_paired(name):
    body = KERNELS[name]
    assert body.count("bcl_arrive(") == body.count("bcl_started(") == 1
    a, b = body.index("bcl_arrive("), body.index("bcl_started(")
    assert a < b and not re.search(r"cl\.sync|bcl_sync|bcl_sums|\breturn\b", re.sub(r"=\s*\[&\].*", "", body[a:b], flags=re.S))
