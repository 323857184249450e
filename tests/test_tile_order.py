"""The walk over a product's output tiles (csrc/tile_order.h, host code): every
tile once, in the order of the bands and groups, for every tile shape, and for
products of more than 65536 row or column blocks; the word that holds a tile."""

import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_13299_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "tile_order.h"
int main(int, char** v) {
  const long long m = atoll(v[1]), n = atoll(v[2]);
  const int bm = atoi(v[3]), bn = atoi(v[4]), sym = atoi(v[5]), units = atoi(v[6]), print = atoi(v[7]);
  dmp::TileOrder order(m, n, bm, bn, sym != 0, units);
  const long long tm = (m + bm - 1) / bm, tn = (n + bn - 1) / bn, count = order.count();
  std::vector<unsigned char> seen(tm * tn, 0);
  long long distinct = 0, outside = 0;
  for (long long i = 0; i < count; ++i) {
    // as the kernels get it
    const dmp::TileAt t = dmp::unpack_tile(dmp::pack_tile(order.next(), order.column_bits()), order.column_bits());
    if (print) printf("%d %d\n", (int)t.bi, (int)t.bj);
    const long long r = t.bi, c = t.bj;
    // symmetric: only tiles holding some element with row <= column
    if (r < 0 || r >= tm || c < 0 || c >= tn || (sym && r * bm >= (c + 1) * bn)) {
      ++outside;
      continue;
    }
    distinct += seen[r * tn + c] == 0;
    seen[r * tn + c] = 1;
  }
  long long want = 0;
  for (long long c = 0; c < tn; ++c)
    for (long long r = 0; r < tm; ++r) want += !sym || r * bm < (c + 1) * bn;
  if (!print) printf("%lld %lld %lld %lld\n", count, distinct, outside, want);
  return 0;
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    d = tmp_path_factory.mktemp("tile_order")
    (d / "walk.cc").write_text(PROGRAM)
    exe = d / "walk"
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(d / "walk.cc"), "-o", str(exe)], check=True)

    def run(*args):
        return subprocess.run([str(exe)] + [str(int(a)) for a in args], check=True, capture_output=True,
                              text=True).stdout

    return run


SHAPES = [(256, 256), (128, 256), (128, 128), (128, 64)]


@pytest.mark.parametrize("bm,bn", SHAPES)
@pytest.mark.parametrize("m,n,sym", [(16_800_000, 64, 0), (64, 16_800_000, 0), (8_400_000, 500, 0), (20000, 20000, 1),
                                     (1, 1, 0), (1, 1, 1), (257, 255, 0), (1000, 1000, 1), (5000, 333, 0)])
def test_every_tile_once(walk, bm, bn, m, n, sym):
    for units in (1, 76, 152):
        count, distinct, outside, want = map(int, walk(m, n, bm, bn, sym, units, 0).split())
        assert (count, distinct, outside) == (want, want, 0)


def _bands(m, n, bm, bn, sym, units):
    """The order written out: bands of w column blocks, groups of h row blocks."""
    tm, tn = -(-m // bm), -(-n // bn)
    w = max(1, min(int((units * bm / bn) ** 0.5 + 0.5), tn))
    h = max(1, units // w)
    rows = lambda c: min(tm, -(-(bn * (c + 1)) // bm)) if sym else tm
    out = []
    for c0 in range(0, tn, w):
        c1 = min(tn, c0 + w)
        for r0 in range(0, rows(c1 - 1), h):
            for c in range(c0, c1):
                out += [(r, c) for r in range(r0, min(rows(c), r0 + h))]
    return out


@pytest.mark.parametrize("bm,bn", SHAPES)
@pytest.mark.parametrize("m,n,sym", [(4096, 4096, 1), (4096, 4096, 0), (3000, 700, 0), (100, 6000, 0), (2305, 2305, 1)])
def test_order_of_the_walk(walk, bm, bn, m, n, sym):
    got = [tuple(map(int, l.split())) for l in walk(m, n, bm, bn, sym, 76, 1).splitlines()]
    assert got == _bands(m, n, bm, bn, sym, 76)


@pytest.mark.parametrize("m,n,sym", [(256 * 3_000_000, 1, 0), (1, 256 * 3_000_000, 0), (2_000_000, 40_000, 0)])
def test_words_of_the_largest_products(walk, m, n, sym):
    """Products whose operands or result fill the GPU's memory."""
    count, distinct, outside, want = map(int, walk(m, n, 256, 256, sym, 76, 0).split())
    assert (count, distinct, outside) == (want, want, 0)
