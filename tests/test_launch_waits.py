"""Kernels of level.cu that are launched before their predecessor has ended (programmatic launch): on
every way out of them stands a wait for it, or what runs after them would start while the
predecessor still writes.  Read from the source (no GPU): the ways out concerned are error paths."""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2408_14193_gb300", "csrc",
                   "level.cu")


def _kernel(name):
    """Body of __global__ function `name` without comments."""
    text = re.sub(r"//[^\n]*", "", open(SRC).read())
    at = re.search(r"__global__[^;{]*\b%s\(" % name, text).end()
    start = text.index("{", at)
    depth, i = 1, start + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        i += 1
    return text[start + 1:i - 1]


def test_sparsify_kernel_has_one_way_out():
    body = _kernel("sparsify_kernel")
    assert not re.search(r"\breturn\b", body)
    assert body.strip().splitlines()[-1].strip() == "if (blockIdx.x == gridDim.x - 1) pdl_wait();"


@pytest.mark.parametrize("name", ["seg_team_kernel", "sep_team_kernel", "seg_solve_kernel", "sep_solve_kernel"])
def test_level_solves_wait_before_each_return(name):
    body = _kernel(name)
    first = re.search(r"^  pdl_wait\(\);", body, re.M)       # the wait that every other thread passes
    assert first
    for m in re.finditer(r"\breturn;", body[:first.start()]):
        assert body[:m.start()].rstrip().endswith("pdl_wait();"), body[max(0, m.start() - 80):m.end()]
