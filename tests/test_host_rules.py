"""The host side's rules, compiled alone from csrc (no GPU needed)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2609_17983_gb300", "csrc")


def run(tmp_path, source):
    """Standard output of a C++ program over the repository's headers, in words."""
    cxx = shutil.which("g++") or pytest.skip("no C++ compiler")
    src, exe = tmp_path / "rule.cpp", tmp_path / "rule"
    src.write_text(source)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-pthread", "-I", CSRC, src,
                    "-o", exe], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()


def test_rows_go_out_by_stores_only_inside_one_writable_range(tmp_path):
    # a page-locked range of 4096 bytes at 0x10000
    out = run(tmp_path, r"""
#include <cstdio>
#include "host_rules.cuh"
using namespace kvr;
int main() {
  const HostRange r{true, true, 0, 0x10000, 4096};
  auto fits = [](uintptr_t p, size_t bytes, HostRange x, uintptr_t shift = 0) {
    x.device = p + shift;
    std::printf("%d ", (int)device_stores_fit(p, bytes, x));
  };
  fits(0x10000, 4096, r);      // all of it
  fits(0x10ff0, 16, r);        // its last bytes
  fits(0x10000, 4097, r);      // one byte past the registration
  fits(0x10ff0, 32, r);        // from its last bytes into a neighbour
  fits(0x10000, (size_t)1 << 34, r);
  fits(0x11000, 16, r);        // behind it
  fits(0xfff0, 16, r);         // before it
  fits(0x10000, ~(size_t)0, r);
  fits(0x10000, 16, r, 4096);  // mapped at another device address
  HostRange x = r;
  x.writable = false;
  fits(0x10000, 16, x);
  x = r;
  x.page_locked = false;
  fits(0x10000, 16, x);
  fits(0x10000, 16, HostRange{});
}
""")
    assert out == ["1", "1"] + ["0"] * 10


def test_settings_are_raised_on_each_device_and_never_lowered(tmp_path):
    out = run(tmp_path, r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "host_rules.cuh"
using namespace kvr;
int main() {
  PerDevice<size_t> s;
  std::vector<std::pair<int, size_t>> calls;
  auto raise = [&](int dev, size_t bytes, int err = 0) {
    const int e = raise_to(s, dev, bytes, [&](size_t b) { calls.push_back({dev, b}); return err; });
    std::printf("%d:%zu ", e, calls.size());
  };
  raise(0, 100);     // set
  raise(0, 100);     // known
  raise(1, 100);     // another device: set there too
  raise(0, 60);      // a smaller request lowers nothing
  raise(2, 100, 7);  // a failure is reported
  raise(2, 100);     // and not remembered
  raise(MAX_DEVICES, 100);
  raise(MAX_DEVICES, 100);
  // threads with different requests: each finds its own granted when it returns
  PerDevice<size_t> t;
  std::atomic<size_t> granted{0};
  std::atomic<int> low{0};
  std::vector<std::thread> th;
  for (size_t i = 1; i <= 8; ++i)
    th.emplace_back([&, i] {
      for (size_t k = 0; k < 2000; ++k) {
        const size_t want = i * 1000 + k;
        raise_to(t, 0, want, [&](size_t b) { granted = b; return 0; });
        if (granted < want) ++low;
      }
    });
  for (auto &x : th) x.join();
  std::printf("%d", low.load());
}
""")
    assert out == ["0:1", "0:1", "0:2", "0:2", "7:3", "0:4", "0:5", "0:6", "0"]


def test_kernels_take_shared_memory_through_that_rule():
    # a process-wide "already set" would leave a model on a second device without it
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        uses = text.count("cudaFuncSetAttribute(")
        assert uses == (1 if name == "kvr_internal.cuh" else 0), name


def test_paired_gemm_waits_only_for_clusters_before_the_waiting_one(tmp_path):
    # every split of a launch's tiles: each unit of K of each tile is computed once,
    # the parts of a tile by clusters in part order, the last of which sums them --
    # one of a higher number than all it waits for, so dispatched after them
    out = run(tmp_path, r"""
#include <cstdio>
#include <map>
#include <vector>
#include "pair_split.cuh"
using namespace kvr;
int main() {
  int checked = 0;
  for (int clusters : {1, 2, 3, 7, 70, 76})
    for (int tiles = 1; tiles <= 3 * clusters; tiles += 1 + clusters / 9)
      for (int KU : {1, 4, 9, 33, 112})
        for (int most = 1; most <= 8; ++most) {
          PairSplit p{KU, 3, clusters, tiles % clusters, 1, tiles / clusters};
          if (p.left) p.parts = clusters / p.left < most ? clusters / p.left : most;
          if (p.parts > KU) p.parts = KU;
          if (!p.rounds) p.clusters = p.left * p.parts;
          std::map<int, std::vector<int>> units;   // of a tile: times computed
          std::map<int, int> sum;                  // of a split tile: its summing cluster
          for (int c = 0; c < p.clusters; ++c) {
            Walk w(p, c);
            Segment s;
            for (bool first = true; w.next(p, s); first = false) {
              auto &u = units[s.tile];
              u.resize(KU);
              for (int k = s.ku0; k < s.ku1; ++k) ++u[k];
              if (s.ku1 - s.ku0 == KU) continue;
              if (!first || s.ntile * 3 + s.mtile != s.tile) return std::puts("order"), 0;
              if (sums_parts(p, c)) {
                if (sum.count(s.tile) || s.ku1 != KU) return std::puts("sums"), 0;
                sum[s.tile] = c;
              }
            }
          }
          if ((int)units.size() != tiles) return std::puts("tiles"), 0;
          for (auto &u : units)
            for (int n : u.second)
              if (n != 1) return std::puts("units"), 0;
          if (p.parts > 1)
            for (int t = 0; t < p.left; ++t)
              for (int k = 0; k < p.parts; ++k) {
                const int c = part_cluster(p, t, k);
                Walk w(p, c);
                Segment s;
                if (!w.next(p, s) || s.tile != t || s.ku0 != k * KU / p.parts)
                  return std::puts("parts"), 0;
                if (!sum.count(t) || (k + 1 < p.parts ? c >= sum[t] : c != sum[t]))
                  return std::puts("waits"), 0;
                ++checked;
              }
        }
  std::puts(checked > 1000 ? "ok" : "few");
}
""")
    assert out == ["ok"]
