"""CPU: index arithmetic of kernels (csrc/kk_walk.h), compiled for the host and
replayed lane by lane: every entry that a lane reads lies inside its array."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2103_11991_gb300 import _build

REPLAY = r"""
#include "kk_walk.h"
using namespace kk;
// The walk of one chunk's products as k_num_chunk does it: pieces (first[k],
// len[k]) of B, in the order of A's row, by `warps` warps and `u` steps a round.
// Returns 0, or 1 + the product whose lane left its piece, or -1 when a product
// was not taken exactly once.
extern "C" int replay(int np, const int* first, const int* len, int warps, int u, int* taken) {
  int start[513], total = 0;
  for (int k = 0; k < np; ++k) { start[k] = total; total += len[k]; }
  start[np] = 0x7fffffff;
  const int threads = warps * 32, per = (total + threads - 1) / threads * 32;
  for (int w = 0; w < warps; ++w) {
    const int f_lo = w * per < total ? w * per : total, f_hi = f_lo + per < total ? f_lo + per : total;
    int seen = 0;
    for (int k = 0; k < np; ++k) seen += start[k] < f_lo;
    for (int f = f_lo; f < f_hi; f += 32 * u)
      for (int s = 0; s < u; ++s) {
        const int fb = f + s * 32;
        uint32_t m = 0;
        for (int lane = 0; lane < 32; ++lane) m |= walk_start_bit(start[seen + lane < np ? seen + lane : np], fb, f_hi);
        for (int lane = 0; lane < 32; ++lane) {
          const int own = seen + __builtin_popcount(m & walk_upto(lane)) - 1;
          const int p = walk_product(fb, lane, f_hi);
          if (own < 0 || own >= np) return 1 + p;
          const int q = first[own] - start[own] + p;
          if (q < first[own] || q >= first[own] + len[own]) return 1 + p;
          if (fb + lane < f_hi) ++taken[p];
        }
        seen += __builtin_popcount(m);
      }
  }
  for (int p = 0; p < total; ++p) if (taken[p] != 1) return -1;
  return 0;
}

// The tiles that CTA `cta` of `ctas` takes of `count` samples; -1 when one begins
// outside them or before the one before.
extern "C" int tiles(int cta, int ctas, int count) {
  int n = 0, last = -1;
  for (int t0 = cta * 32; t0 < count; t0 = walk_next_tile(t0, ctas * 32, count)) {
    if (t0 <= last) return -1;
    last = t0;
    ++n;
  }
  return n;
}
"""


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    d = tmp_path_factory.mktemp("walk")
    src, lib = d / "walk.cpp", d / "walk.so"
    src.write_text(REPLAY)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", _build.CSRC, str(src), "-o", str(lib)],
                   check=True)
    return ctypes.CDLL(os.fspath(lib))


def _walk(lib, first, lens, u):
    a, b = np.asarray(first, np.int32), np.asarray(lens, np.int32)
    taken = np.zeros(max(1, int(b.sum())), np.int32)
    return lib.replay(len(b), *(x.ctypes.data_as(ctypes.c_void_p) for x in (a, b)), 8, u,
                      taken.ctypes.data_as(ctypes.c_void_p))


@pytest.mark.parametrize("order", ["as drawn", "descending", "repeated"])
@pytest.mark.parametrize("high", [1, 3, 40, 200, 700])
def test_lanes_past_a_run_stay_in_its_pieces(replay, order, high):
    # pieces of A rows in no order: entries of B that begin anywhere, its first among them
    rng = np.random.RandomState(high)
    assert _walk(replay, [60, 0], [40, 60], 2) == 0  # one step whose second one lies past the run
    for _ in range(60):
        lens = rng.randint(1, high + 1, rng.randint(1, 257))
        first = rng.permutation(np.cumsum(lens) - lens) if order == "as drawn" else \
            np.cumsum(lens[::-1])[::-1] - lens if order == "descending" else np.zeros(len(lens), int)
        for u in (1, 2, 4):
            assert _walk(replay, first, lens, u) == 0


@pytest.mark.parametrize("count", [1, 32, 33, 19456, 19457, 2 ** 31 - 19457, 2 ** 31 - 19456, 2 ** 31 - 1])
def test_tiles_of_samples_end(replay, count):
    for ctas in (8, 608):
        got = [replay.tiles(c, ctas, count) for c in (0, 1, ctas - 1)]
        assert got == [max(0, -(-(-(-count // 32) - c) // ctas)) for c in (0, 1, ctas - 1)]
