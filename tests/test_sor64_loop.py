"""Checks, launch lengths and exchange numbers of the FP64 solve kept on chip
(csrc/sor64_loop.h), compiled for the host: the launches of a solve together
check where one loop over its sweeps would (before the first and every m, at
most maxs sweeps), none is longer than its limit whatever m is, and none uses
more exchange numbers than it reserves.  The exchanges are counted as
k_sor64_tiles makes them: a halo of K cells lasts K half-sweeps, a check needs
one half-sweep's worth of it, a sweep two."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2402_17337_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "sor64_loop.h"
using namespace ibm;
#define REQUIRE(x) do { if (!(x)) { std::printf("%s: m %d maxs %d chunk %d K %d converges %d\n", #x, m, maxs, chunk, K, conv); std::exit(1); } } while (0)

// the sweep counts at which a solve checks, and how it ends; conv: the check that meets the tolerance (-1: none)
static void reference(int m, int maxs, int conv, std::vector<long long>& at, int& status, long long& sweeps) {
  for (long long s = 0;; ++s) {
    if (s % m == 0) {
      at.push_back(s);
      if ((int)at.size() - 1 == conv) { status = SOR64_OK; sweeps = s; return; }
    }
    if (s >= maxs) { status = SOR64_NOCONV; sweeps = s; return; }
  }
}

static void solve(int m, int maxs, int chunk, int K, int conv) {
  std::vector<long long> want, got;
  int status = 0, launches = 0;
  long long sweeps = 0;
  reference(m, maxs, conv, want, status, sweeps);
  Sor64Progress run{m, maxs, chunk};
  unsigned used = 0;
  for (;;) {
    const unsigned before = used;
    unsigned first = 0;
    REQUIRE(!sor64_reserve(&used, &first) && first == before && used - before == kSor64Numbers);
    const Sor64Span span = run.span();
    Sor64Loop L(span);
    unsigned no = first;
    int fresh = K;
    for (;;) {
      if (L.check_due()) {
        if (fresh < 1) { ++no; fresh = K; }
        ++no;
        got.push_back(run.done + L.s);
        if (L.checked(span, got.size(), true, (int)got.size() - 1 == conv)) break;
      }
      if (L.stop(span)) break;
      if (fresh < 2) { ++no; fresh = K; }
      fresh -= 2;
      ++L.s;
    }
    ++launches;
    REQUIRE(L.s <= chunk);
    REQUIRE(no - first <= kSor64Numbers);
    REQUIRE(L.last < 0 || L.bits == got.size());
    run.advance(L.s, L.last);
    if (L.status != SOR64_MORE) {
      REQUIRE(L.status == status && run.done == sweeps);
      break;
    }
    REQUIRE(L.s == chunk);
  }
  REQUIRE(launches <= sweeps / chunk + 1);
  REQUIRE(got == want);
}

int main() {
  const int ms[] = {1, 2, 3, 7, 8, 100, 1023, 1024, 1025, 8191, 8192, 8193, 16384, 65536, 65537, 65538, 65539, 2147483647};
  const int maxs[] = {0, 1, 2, 7, 8, 60, 1024, 1025, 8192, 8193, 20000, 140000};
  for (int m : ms)
    for (int mx : maxs)
      for (int chunk : {1, 5, kSor64TilesChunk, kSor64Chunk})
        for (int K = 2; K <= 8; K += 2)
          for (int conv : {-1, 0, 1, 3})
            if (chunk > 5 || mx <= 8192) solve(m, mx, chunk, K, conv);
  // the limit of the counts themselves
  Sor64Progress run{2147483647, 2147483647, kSor64Chunk};
  run.advance(0, 0);
  run.done = 2147483600ll;
  const Sor64Span p = run.span();
  if (p.next != 47 || p.maxs != 47) return 2;
  // numbers run out: start again, and say so
  unsigned used = 4294967295u - kSor64Numbers, first = 0;
  if (sor64_reserve(&used, &first) || first != 4294967295u - kSor64Numbers || used != 4294967295u) return 3;
  if (!sor64_reserve(&used, &first) || first != 0 || used != kSor64Numbers) return 4;
  return 0;
}
"""


def test_launches_check_end_and_number_as_one_loop_would(tmp_path):
    cxx = os.environ.get("CXX") or shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "loop.cpp", tmp_path / "loop"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, (out.returncode, out.stdout)
