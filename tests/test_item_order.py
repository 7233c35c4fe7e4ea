"""The order of a sequence's work items (csrc/item_order.h), compiled for the host: every (head, block) comes up exactly once,
and under a causal mask the blocks of a group of heads come heaviest first."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_07524_b200", "csrc")
WRAPPER = """
#include "item_order.h"
extern "C" void places(uint32_t nblk, uint32_t heads, uint32_t workers, int causal, int heavy_is_last, uint32_t* out) {
    for (uint32_t i = 0; i < nblk * heads; ++i) {
        const dcp::ItemPlace p = dcp::item_place(i, nblk, heads, workers, causal != 0, heavy_is_last != 0);
        out[2 * i] = p.head;
        out[2 * i + 1] = p.blk;
    }
}
"""


@pytest.fixture(scope="module")
def places(tmp_path_factory):
    d = tmp_path_factory.mktemp("item_order")
    src, so = str(d / "places.cpp"), str(d / "places.so")
    with open(src, "w") as f:
        f.write(WRAPPER)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    fn = ctypes.CDLL(so).places

    def call(nblk, heads, workers, causal, heavy_is_last):
        out = np.empty((nblk * heads, 2), dtype=np.uint32)
        fn(nblk, heads, workers, int(causal), int(heavy_is_last), out.ctypes.data_as(ctypes.c_void_p))
        return out.astype(np.int64)
    return call


@pytest.mark.parametrize("workers", [1, 2, 74, 148])
@pytest.mark.parametrize("causal,heavy_is_last", [(False, False), (True, False), (True, True)])
def test_every_head_and_block_comes_up_once(places, workers, causal, heavy_is_last):
    uneven = 0
    for heads in (1, 2, 3, 4, 5, 7, 8, 12, 16, 31):
        for nblk in (1, 2, 3, 5, 8, 37, 62, 75, 100, 148, 149, 297, 512):
            p = places(nblk, heads, workers, causal, heavy_is_last)
            assert p[:, 0].max() < heads and p[:, 1].max() < nblk
            assert np.unique(p[:, 0] * nblk + p[:, 1]).size == nblk * heads, (heads, nblk)
            least = -(-2 * workers // nblk)
            uneven += causal and least < heads and heads % (heads // least) != 0
    assert not causal or uneven >= 5 or workers < 74          # groups of unequal size are among them


@pytest.mark.parametrize("heavy_is_last", [False, True])
def test_causal_groups_are_whole_heads_heaviest_block_first(places, heavy_is_last):
    for heads, nblk, workers in ((4, 62, 74), (16, 32, 148), (16, 100, 74), (7, 75, 148), (8, 512, 148), (3, 5, 148)):
        p = places(nblk, heads, workers, True, heavy_is_last)
        least = -(-2 * workers // nblk)
        i, seen = 0, 0
        while i < len(p):
            # a group: the first block of its heads, one after the other, then the next block of the same heads
            first = nblk - 1 if heavy_is_last else 0
            size = 1
            while i + size < len(p) and p[i + size, 1] == first and p[i + size, 0] == p[i, 0] + size:
                size += 1
            group = p[i:i + size * nblk]
            assert (group[:, 0].reshape(nblk, size) == np.arange(seen, seen + size)).all()
            order = np.arange(nblk)[::-1] if heavy_is_last else np.arange(nblk)
            assert (group[:, 1].reshape(nblk, size) == order[:, None]).all()
            assert size >= min(least, heads)
            seen += size
            i += size * nblk
        assert seen == heads
