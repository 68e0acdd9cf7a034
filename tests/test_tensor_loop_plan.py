"""The plans of the resident-factor launch (k_tensor_loop.cu) over its whole
range of shapes: tensor-memory columns, shared memory, segments, grid and
counters within their limits (CPU; a program linked against the library calls
the rule itself)."""
import glob
import os
import shutil
import subprocess

import pytest

import paper_1905_00689_gb300 as package
from paper_1905_00689_gb300 import _binding

CSRC = os.path.join(os.path.dirname(package.__file__), "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "internal.h"
using namespace lstm_approx_impl;

static Checkpoints depths(int K, unsigned* seed) {
  Checkpoints c{};
  auto next = [&](int n) { return (int)((*seed = *seed * 1664525u + 1013904223u) >> 8) % n; };
  const int want = next(kMaxCheckpoints + 1);
  for (int i = 0, at = 0; i < want && at < K; ++i) {
    at += 1 + next(i % 2 ? 16 : (K + want - 1) / want);
    if (next(2)) at = (at + 15) / 16 * 16;
    if (at > K) break;
    c.k[c.n++] = at;
  }
  return c;
}

#define CHECK(x) do { if (!(x)) { std::printf("H %d B %d K %d J %d: %s\n", H, B, K, ck.n, #x); std::exit(1); } } while (0)

int main() {
  long plans = 0, splits = 0, shared = 0, streamed = 0;
  unsigned seed = 7;
  const int Hs[] = {1, 63, 64, 65, 127, 128, 129, 301, 512, 513, 640, 1000, 1024, 1025, 1100, 1536, 2047, 2048};
  const int Ks[] = {1, 15, 16, 17, 32, 33, 64, 65, 90, 127, 128, 129, 200, 255, 256, 300, 512, 513, 640, 800, 902, 1000, 1023, 1024};
  const int Bs[] = {1, 2, 15, 16, 17, 31, 32, 33, 64, 65, 100, 128, 256, 300, 511, 700, 1024, 2000, 4096};
  for (int H : Hs) for (int K : Ks) for (int B : Bs) for (int rep = 0; rep < 12; ++rep) for (bool slower_too : {false, true}) {
    Checkpoints ck = rep == 0 ? Checkpoints{} : depths(K, &seed);
    TcLoopPlan p;
    if (!tc_loop_plan(H, B, K, ck, slower_too, &p)) continue;
    ++plans;
    const int gb = 4 / p.gp, nkb = (K + 63) / 64, nsl = (K + 15) / 16;
    CHECK(p.nt == 16 || p.nt == 32);
    CHECK(p.gp == 4 || p.gp == 1);
    // the grid: whole clusters, at most one wave, every stream tile in both roles
    CHECK(p.cs == (p.ga > gb ? p.ga : gb) && p.cs % p.ga == 0 && p.cs % gb == 0);
    CHECK(p.ctas % p.cs == 0 && p.ctas <= (p.cs == 4 ? 144 : 148) && p.nA <= p.ctas && p.nB <= p.ctas);
    CHECK(p.ST * p.nt >= B && (p.ST - 1) * p.nt < B && p.ST <= kLoopMaxTiles);
    CHECK(p.nA == p.RT * p.ga * ((p.ST + p.sa - 1) / p.sa) && p.nB == p.UT * gb * ((p.ST + p.sb - 1) / p.sb));
    CHECK(p.UT * 128 >= H && p.ga * p.nka * 64 >= H && p.nka <= 8);
    CHECK(p.rpg == 128 ? p.RT == 4 * p.ktiles && p.ktiles * 128 >= K : p.RT * 128 / p.rpg >= 4 && p.rpg >= K);
    // the segments: ascending, one ending at each depth below K, whole slices elsewhere
    int ndep = 0, pieces = 0, last_split = -1;
    while (ndep < ck.n && ck.k[ndep] < K) {
      if (ck.k[ndep] % 16) { ++pieces; last_split = ck.k[ndep] / 16; }
      ++ndep;
    }
    CHECK(p.ndep == ndep && p.ncut >= ndep && p.ncut <= kLoopMaxCuts && p.split_depths == (pieces > 0));
    for (int i = 0, d = 0; i < p.ncut; ++i) {
      const int lo = i ? p.cut_k[i - 1] : 0;
      CHECK(p.cut_k[i] > lo && p.cut_k[i] < K);
      if (d < ndep && p.cut_k[i] == ck.k[d]) { CHECK(p.dep_segs[d] == i + 1); ++d; }
      else CHECK(p.cut_k[i] % 16 == 0);
      if (K > 512) CHECK(p.cut_k[i] - lo <= kLoopSegTerms + 16);
      if (i == p.ncut - 1) CHECK(d == ndep && (K <= 512 || K - p.cut_k[i] <= kLoopSegTerms + 16));
    }
    CHECK(p.stream_segs == (p.ncut > 0 && ndep == 0));
    // tensor memory: U, then either role's accumulators, in 512 columns
    const int slices = 4 * p.ures < nsl ? 4 * p.ures : nsl;
    const int seg = (p.stream_segs ? 1 : p.ncut + 1) * p.gp * p.nt * (1 + p.mb);
    CHECK(last_split < slices);
    CHECK((slices + pieces) * p.gp * 8 <= p.acc_a && p.acc_a % 32 == 0);
    CHECK(p.ra_regions >= 1 && p.ra_regions <= 4 && p.rb_regions >= 1 && p.rb_regions <= 4);
    CHECK(p.acc_a + p.ra_regions * 2 * p.nt <= (p.shared_acc ? 512 : p.acc_b));
    CHECK(p.shared_acc ? p.acc_b == p.acc_a : p.acc_b > p.acc_a);
    CHECK(p.acc_b + p.rb_regions * seg <= 512);
    CHECK(!p.defer_depths || (ndep > 0 && !p.shared_acc && p.rb_regions >= p.sb));
    // shared memory: factors, ring, receive buffers, barriers
    CHECK(p.ux_chunks == p.gp * (nkb - p.ures) && p.ures >= 0 && p.ures <= nkb);
    CHECK(p.rxa_bytes == (p.ga > 1 ? 128u * p.nt * 4 : 0u) && p.rxb_bytes == (gb > 1 ? 4u * 128 * (p.nt / gb) * 4 : 0u));
    const unsigned rx = p.share_rx ? 2 * (p.rxa_bytes > p.rxb_bytes ? p.rxa_bytes : p.rxb_bytes) : 2 * (p.rxa_bytes + p.rxb_bytes);
    CHECK(p.stages >= p.gp && p.stages <= 16 && p.stages * p.nt >= 128);
    CHECK(16384u * (p.nka + p.ux_chunks) + p.stages * p.nt * 256u + rx + 1024u + 1024u <= p.smem && p.smem <= 227u * 1024);
    splits += pieces > 0;
    shared += p.shared_acc;
    streamed += p.stream_segs;
  }
  std::printf("%ld plans, %ld split, %ld shared, %ld streamed\n", plans, splits, shared, streamed);
  return plans > 10000 && splits > 1000 && shared > 0 && streamed > 100 ? 0 : 1;
}
"""


def test_plans_stay_within_their_limits(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    includes = [p for p in [os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include"),
                            *glob.glob("/usr/local/cuda*/include")] if os.path.exists(os.path.join(p, "cuda_runtime.h"))]
    if not includes:
        pytest.skip("no CUDA headers")
    _binding.load()
    (tmp_path / "p.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-I", includes[0], str(tmp_path / "p.cpp"), _binding.LIB_PATH,
                    "-Wl,-rpath," + os.path.dirname(_binding.LIB_PATH), "-o", str(tmp_path / "p")], check=True)
    r = subprocess.run([str(tmp_path / "p")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
