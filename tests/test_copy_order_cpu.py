"""Copies out of shared memory are issued by one lane for bytes that other threads wrote: between the writers' proxy fence and the copy stands a
barrier of those threads.  A missing one cannot be made to fail by running (a converged warp issues in order), so the sources are read."""
import os
import re

import pytest

from paper_2203_16487_b200 import build

COPY = re.compile(r"cp\.async\.bulk(\.tensor)?[.\w:]*\.(shared::cluster|global)\.(tile\.)?shared::cta")
BARRIER = re.compile(r"__syncwarp\(\)|__syncthreads\(\)|\bbar\.sync\b|\btc_cluster_sync\(\)")


def _copies():
    for path in build.SOURCES + build.HEADERS:
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in COPY.finditer(text):
            yield os.path.basename(path), text[:m.start()]


def test_the_copies_are_found():
    assert {name for name, _ in _copies()} >= {"attention.cuh", "gemm_tc_splitk.cuh"}


@pytest.mark.parametrize("name,before", list(_copies()), ids=lambda v: v if v.endswith(".cuh") else "")
def test_a_barrier_between_the_fence_and_the_copy(name, before):
    fence = before.rfind("fence.proxy.async")
    assert fence >= 0, name
    assert BARRIER.search(before, fence), f"{name}: a lane copies what other lanes wrote, nothing orders it behind their stores"
