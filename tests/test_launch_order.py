"""Kernels that take tensor memory let the next grid start only once they have it, read from their sources: the call comes from the
allocating warp after the allocation, or behind a block-wide barrier after it (the reason stands at `grid_dependency_wait`)."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2212_01005_b200", "csrc")
ALLOC = re.compile(r"if \((warp == [^)]+)\) \{\s*(tmem_alloc(?:_pair)?\([^;]*;[^}]*)\}")
LAUNCH = re.compile(r"grid_launch_dependents(?:\(\)|_if\((warp == [^)]+)\));")


def kernels():
    """(file, body) of every kernel with an allocation: from its `__global__` to the next one."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for body in re.split(r"(?=__global__)", text)[1:]:
            if "tmem_alloc" in body:
                yield os.path.basename(path), body


def in_order(body):
    allocs = ALLOC.findall(body)
    assert len(allocs) == 1 and len(re.findall(r"\btmem_alloc(?:_pair)?\(", body)) == 1
    (warp, block), at = allocs[0], ALLOC.search(body)
    for m in LAUNCH.finditer(body):
        own = at.start() < m.start() < at.end()                                     # in the allocating branch, after the call
        barrier = re.search(r"\n  __syncthreads\(\);", body[at.end():m.start()]) if m.start() > at.end() else None
        if not (own and body[at.start():m.start()].find("tmem_alloc") >= 0) and not barrier and not (m.start() > at.end() and m.group(1) == warp):
            return False
    return True


def test_next_grid_starts_after_the_allocation():
    found = [(f, in_order(b)) for f, b in kernels()]
    assert len(found) >= 9
    assert all(ok for _, ok in found), found


@pytest.mark.parametrize("body, ok", [
    ("__global__ if (warp == 0) { tmem_alloc(s, 512); } grid_launch_dependents();\n  __syncthreads();", False),
    ("__global__ grid_launch_dependents(); if (warp == 0) { tmem_alloc(s, 512); }\n  __syncthreads();", False),
    ("__global__ if (warp == 0) { tmem_alloc(s, 512); } grid_launch_dependents_if(warp == 1);\n  __syncthreads();", False),
    ("__global__ if (warp == 0) { tmem_alloc(s, 512); } grid_launch_dependents_if(warp == 0);\n  __syncthreads();", True),
    ("__global__ if (warp == 0) { tmem_alloc(s, 512); }\n  __syncthreads(); grid_launch_dependents();", True),
])
def test_orders_that_are_told_apart(body, ok):
    assert in_order(body) == ok
