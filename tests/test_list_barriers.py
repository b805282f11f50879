"""The list kernels clear a table of their warp in shared memory, each lane a
part of it, and fill it from any lane: a warp barrier has to lie between, or a
lane's entry can be erased by another lane's later clearing (a lost entry is an
exclusion that is not applied).  Today's compiler keeps such a warp together,
so no run shows a missing barrier; the source does."""

import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_0902_0827_gb300", "csrc",
                   "nb_build.cu")


def kernel_body(name):
    src = re.sub(r"//[^\n]*", "", open(SRC).read())
    m = re.search(r"__global__[^;{]*\b" + name + r"\([^)]*\)\s*\{", src)
    assert m, name
    depth, k = 1, m.end()
    while depth:
        depth += {"{": 1, "}": -1}.get(src[k], 0)
        k += 1
    return src[m.end():k]


@pytest.mark.parametrize("kernel,clear,fill", [("k_glist", "s_head_all[w][t] = kLinkEnd", "hset_insert("),
                                               ("k_glist1", "s_map[lane] = 0u", "atomicOr(&s_map")])
def test_barrier_between_clearing_and_filling(kernel, clear, fill):
    body = kernel_body(kernel)
    cleared, filled = body.index(clear), body.index(fill)
    assert cleared < filled
    assert "__syncwarp()" in body[cleared:filled]
