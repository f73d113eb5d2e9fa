"""The host side's rules, compiled alone from csrc/host_rules.cuh (no GPU needed)."""
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
