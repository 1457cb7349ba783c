"""Hub rows of the source kernel cut into pieces (csrc/pieces.h, source.cu).

A step lists up to 64 rows of more than 512 arcs but counts the pieces of all of
them, so the last row listed is asked for piece numbers far past its own.  On the
CPU the header's arithmetic is compiled with the host compiler and followed over
whole steps, up to 2^32 - 1 pieces: every arc of a listed row is covered once, and
no piece reaches outside its row.  On the GPU: steps with more long rows than the
list holds, replayed by MFBr's pull (more DAG arcs than are recorded), against the
CPU oracle.
"""
import subprocess

import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1609_07008_gb300 as mfbc
from paper_1609_07008_gb300 import build as mbuild

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "pieces.h"
using namespace mfbc;

static void fail(const char* what, long long a, long long b, long long i) {
  std::printf("%s: row of %lld + %lld arcs, piece %lld\n", what, a, b, i);
  std::exit(1);
}
// pieces i of one row: inside it, in order and complete; none past them
static void row(int32_t out, int32_t in) {
  const uint32_t np = src_pieces(out) + src_pieces(in);
  int64_t at[2] = {0, 0};
  for (uint32_t i = 0; i < np; i++) {
    const HubPiece p = src_hub_piece(out, in, i);
    if (p.count < 1 || p.count > SRC_PIECE || p.first != at[p.in]) fail("gap", out, in, i);
    at[p.in] += p.count;
  }
  if (at[0] != out || at[1] != in) fail("incomplete", out, in, np);
  for (int s = 0; s < 32; s++)
    for (int64_t d = -3; d <= 3; d++) {
      const int64_t i = (1ll << s) + d;
      if (i >= np && i <= 0xffffffffll && src_hub_piece(out, in, (uint32_t)i).count) fail("past the row", out, in, i);
    }
  if (src_hub_piece(out, in, 0xffffffffu).count) fail("past the row", out, in, 0xffffffffll);
}
// a step: 64 rows listed, the pieces of `more` further rows counted behind them
static void step(int32_t out, int32_t in, uint64_t more) {
  const uint32_t each = src_pieces(out) + src_pieces(in);
  const uint64_t np = (64 + more) * each;
  uint64_t arcs = 0;
  for (uint64_t p = 0; p < np; p++) {
    const uint64_t h = p / each < 64 ? p / each : 63;
    const HubPiece x = src_hub_piece(out, in, (uint32_t)(p - h * each));
    if (x.count && (x.first < 0 || (int64_t)x.first + x.count > (x.in ? in : out))) fail("outside", out, in, (long long)p);
    arcs += (uint64_t)x.count;
  }
  if (arcs != 64ull * ((uint64_t)out + in)) fail("not once", out, in, (long long)arcs);
}
int main() {
  const int32_t lens[] = {0, 1, 255, 256, 257, 512, 513, 1000, 65537, 33554431, 2147483647};
  for (int32_t out : lens)
    for (int32_t in : lens) row(out, in);
  step(513, 0, 100);
  step(600, 700, 1000);
  step(513, 0, 20000000);              // 6 * 10^7 pieces: offsets past 2^31 arcs
  step(40000, 40000, 100000);
  std::puts("ok");
}
"""


def test_pieces_cover_listed_rows_and_nothing_else(tmp_path):
    src, exe = tmp_path / "pieces.cpp", tmp_path / "pieces"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-Wall", "-I", mbuild.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("directed", [False, True])
@pytest.mark.parametrize("weights", [None, (1, 2)])
def test_more_long_rows_than_the_list_holds_in_both_directions(directed, weights):
    mbuild.build()
    mfbc.load()
    g = gg.erdos_renyi(1300, 1200, directed=directed, weights=weights, seed=41)
    srcs = np.array([0, 7, 1299, 640], np.int32)
    G = mfbc.Graph.from_csr(g)
    path = mfbc.PATH_SMALL if weights is None else mfbc.PATH_DIST
    try:
        lam, want = G.bc(srcs, path=path), oracle.bc(g, srcs)
        assert np.array_equal(lam == 0, want == 0)
        assert np.max(np.abs(lam - want)[want != 0] / want[want != 0]) <= 1e-9
        d, s = G.sssp(srcs, path=path)
        wd, ws, _ = oracle.sssp(g, srcs)
        assert np.array_equal(d, wd) and np.array_equal(s, ws)
    finally:
        G.close()
