"""The buffers that the Q tile and the K ring of the attention kernel share, run on the host: the producer's and the issuer's
walks agree, and a buffer is filled again only after the last product that reads what it holds.  Compiled from the kernel's
own header."""
import ctypes
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_32197_b200", "csrc")
SOURCE = """
#include "item_queue.cuh"
// Buffer and parity of every tile of n items: out[2k], out[2k + 1], an item's Q tile before its K tiles.
template <int kRing> static void walk(int n, const int* tiles, int* out) {
  sparsp::QKRing<kRing> at;
  for (int i = 0; i < n; ++i)
    for (int t = -1; t < tiles[i]; ++t) {
      const uint32_t b = t < 0 ? at.next_q() : at.next_k();
      *out++ = (int)b;
      *out++ = (int)at.use(b);
    }
}
extern "C" void walk3(int n, const int* tiles, int* out) { walk<3>(n, tiles, out); }
extern "C" void walk4(int n, const int* tiles, int* out) { walk<4>(n, tiles, out); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("qk_ring")
    src, out = str(d / "ring.cpp"), str(d / "ring.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, src, "-o", out], check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("ring", [3, 4])
@pytest.mark.parametrize("longest", [1, 2, 3, 4, 5, 9, 40])
def test_a_buffer_is_filled_after_its_last_use(lib, ring, longest):
    for seed in range(20):
        rng = random.Random(seed)
        tiles = [rng.randint(1, longest) for _ in range(60)]
        loads = sum(tiles) + len(tiles)
        out = (ctypes.c_int * (2 * loads))()
        getattr(lib, "walk%d" % ring)(len(tiles), (ctypes.c_int * len(tiles))(*tiles), out)
        # products are numbered through; a K tile is read by one of them, a Q tile by all of its item
        held_until, uses, k, product, before = {}, {}, 0, 0, 0
        for n in tiles:
            first, last = product, product + n - 1
            for t in range(-1, n):
                b, parity = out[2 * k], out[2 * k + 1]
                k += 1
                assert 0 <= b <= ring and parity == uses.get(b, 0) % 2
                uses[b] = uses.get(b, 0) + 1
                needed = first if t < 0 else first + t  # the first product that reads this tile
                # what the buffer held has been read by then, so neither side waits for itself ...
                assert held_until.get(b, -1) < needed
                # ... and where lists are long a K tile is on its way ring products ahead (ring - 1 behind a Q tile that
                # took a buffer)
                if t >= 0 and b in held_until and min(n, before) >= ring:
                    assert needed - held_until[b] >= ring - 1
                held_until[b] = last if t < 0 else needed
            product, before = product + n, n
