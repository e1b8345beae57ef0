"""The walk over the attention kernel's work items, run on the host: several CTAs take numbers from one counter in arbitrary
order.  Compiled from the kernel's own header."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_32197_b200", "csrc")
SOURCE = """
#include <algorithm>
#include "item_queue.cuh"
// One claim of CTA `cta` (its first one if first is set), told to give up searching if stop is set.  Returns head * per_head + place, or -1.
extern "C" int claim(int cta, int first, int grid, int per_head, int n_heads, const int32_t* n_items, int* counter, int stop) {
  int x = 0;
  const int it = first ? cta : grid + (*counter)++;
  auto next = [&](int number) {
    *counter = std::max(*counter, std::max(number - grid, 0));
    return grid + (*counter)++;
  };
  const int head = sparsp::find_item(it, per_head, n_heads, n_items, next, [&] { return stop != 0; }, &x);
  return head < n_heads ? head * per_head + x : -1;
}
"""


@pytest.fixture(scope="module")
def claim(tmp_path_factory):
    d = tmp_path_factory.mktemp("item_queue")
    src, lib = str(d / "queue.cpp"), str(d / "queue.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib], check=True)
    fn = ctypes.CDLL(lib).claim

    def call(cta, first, grid, per_head, n_items, counter, stop):
        return fn(cta, first, grid, per_head, len(n_items), n_items.ctypes.data_as(ctypes.c_void_p), ctypes.byref(counter),
                  stop)
    return call


def _heads(rng, n_heads, per_head, kind):
    n = rng.integers(0, per_head + 1, n_heads) if kind == "some" else np.full(n_heads, per_head if kind == "all" else 0)
    return n.astype(np.int32)


@pytest.mark.parametrize("grid,per_head,n_heads", [(1, 1, 1), (4, 9, 3), (148, 7, 40), (148, 300, 2), (148, 12, 5)])
@pytest.mark.parametrize("kind", ["some", "all", "none"])
def test_every_item_is_taken_once(claim, grid, per_head, n_heads, kind):
    for seed in range(20):
        rng = np.random.default_rng(seed)
        n_items = _heads(rng, n_heads, per_head, kind)
        counter, taken, first = ctypes.c_int(0), [], [True] * grid
        running = list(range(min(grid, n_heads * per_head)))
        while running:
            cta = running[rng.integers(len(running))]
            got = claim(cta, first[cta], grid, per_head, n_items, counter, 0)
            first[cta] = False
            if got < 0:
                running.remove(cta)
            else:
                taken.append(got)
        assert sorted(taken) == [h * per_head + x for h in range(n_heads) for x in range(n_items[h])]


@pytest.mark.parametrize("kind", ["some", "none"])
def test_a_stopped_search_returns_an_item_or_nothing(claim, kind):
    """A CTA that gives up while it searches (a wait of it has run out) takes no place behind a head's last item."""
    grid, per_head, n_heads = 5, 8, 6
    for seed in range(50):
        rng = np.random.default_rng(seed)
        n_items = _heads(rng, n_heads, per_head, kind)
        for cta in range(grid):
            counter = ctypes.c_int(int(rng.integers(0, n_heads * per_head)))
            got = claim(cta, int(rng.integers(2)), grid, per_head, n_items, counter, 1)
            assert got == -1 or got % per_head < n_items[got // per_head]
