"""The cuts of a ragged launch (csrc/ragged_cuts.h), compiled for the host: every
block of every warp-group is taken once, a warp-group by two clock warps at
most, and no tail piece comes to its hand-off long before the head is done."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1909_04750_gb300", "csrc")

SRC = r"""
#include "ragged_cuts.h"
using namespace mickey;
// Pieces as rows (slot, warp-group, first block, end); returns their number.
extern "C" long pieces(const uint64_t *c, uint32_t W, uint32_t slots, int tails_first, uint64_t *order,
                       uint64_t *blocks, uint64_t *out, long room) {
  const RaggedLine q = ragged_cuts(c, W, slots, order, blocks);
  long n = 0;
  for (uint32_t s = 0; s < slots; ++s) {
    uint32_t p;
    uint64_t a, b;
    for (uint32_t k = 0; ragged_piece(q, tails_first, s, k, p, a, b); ++k) {
      if (n == room) return -1;
      out[4 * n] = s, out[4 * n + 1] = q.order[p], out[4 * n + 2] = a, out[4 * n + 3] = b;
      ++n;
    }
  }
  return n;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("cuts")
    (d / "cuts.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "cuts.cpp"),
                    "-o", str(d / "cuts.so")], check=True)
    return ctypes.CDLL(str(d / "cuts.so"))


def _pieces(lib, c, slots, tails_first=0):
    c = np.ascontiguousarray(c, np.uint64)
    W, room = len(c), 2 * len(c) + 2 * slots
    order, blocks = np.zeros(W, np.uint64), np.zeros(W + 1, np.uint64)
    out = np.zeros((room, 4), np.uint64)
    lib.pieces.restype = ctypes.c_long
    n = lib.pieces(*(ctypes.c_void_p(c.ctypes.data), ctypes.c_uint32(W), ctypes.c_uint32(slots),
                     ctypes.c_int(tails_first)), *(ctypes.c_void_p(a.ctypes.data)
                                                   for a in (order, blocks, out)),
                   ctypes.c_long(room))
    assert n >= 0
    return out[:n].astype(np.int64)


def _longest_wait(pieces, c):
    """How long, in blocks, the tail pieces wait when every clock warp takes the
    same time per block; heads come first, so none of them waits."""
    done, waits = {}, []
    clock = {}
    for s, w, a, b in pieces:                       # heads and whole warp-groups
        if a == 0:
            clock[s] = clock.get(s, 0) + b
            if b < c[w]:
                done[w] = clock[s]
    for s, w, a, b in pieces:
        if a > 0:
            waits.append(done[w] - clock.get(s, 0))
    return max(waits, default=0)


def _cases():
    rng = np.random.default_rng(2)
    one = np.full(1024, 64)
    one[1] = 1 << 20                                # one stream of 2^27 bits among 2^13
    last = np.full(1024, 64)
    last[1023] = 1 << 27                            # ... of 2^34, in the last warp-group
    few = np.full(1024, 64)
    few[rng.integers(0, 1024, 50)] = 1 << 18
    yield from (one, last, few, np.full(1024, 128), np.full(609, 1), np.full(608, 7),
                rng.integers(64, 129, 1024), rng.integers(0, 3, 5000),
                (2.0 ** rng.uniform(0, 20, 2000)).astype(np.int64),
                np.where(rng.random(3000) < 0.9, 0, rng.integers(0, 1 << 16, 3000)))
    geo = np.zeros(700, np.int64)
    geo[:40] = 1 << np.arange(40)                   # every share is passed again by the next
    yield geo


@pytest.mark.parametrize("slots", [1, 4, 608])
def test_every_block_once_and_no_long_wait(lib, slots):
    for c in _cases():
        pieces = _pieces(lib, c, slots)
        assert np.array_equal(np.sort(_pieces(lib, c, slots, 1), axis=0), np.sort(pieces, axis=0))
        taken = {}
        for s, w, a, b in pieces:
            assert 0 <= a <= b <= c[w]
            taken.setdefault(w, []).append((a, b, s))
        for w in range(len(c)):
            parts = sorted(p for p in taken.get(w, []) if p[0] < p[1])
            assert len(parts) <= 2
            assert sum(b - a for a, b, _ in parts) == c[w]
            assert not parts or (parts[0][0] == 0 and parts[-1][1] == c[w])
            if len(parts) == 2:                     # head, then tail on the next clock warp
                assert parts[0][1] == parts[1][0] and parts[1][2] == parts[0][2] + 1
        assert _longest_wait(pieces, c) <= slots
        # no clock warp has more than the longest warp-group or the even share,
        # rounded up
        load = np.zeros(slots, np.int64)
        for s, w, a, b in pieces:
            load[s] += b - a
        assert load.max() <= max(int(c.max()), -(-int(c.sum()) // slots))
