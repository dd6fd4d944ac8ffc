"""The producer of the tail product (csrc/qg_split_feed.h) on the CPU with each of its waits running out in
turn: every copy requested has landed (its buffer was given back by the consumer) or is waited for before the
block may exit, and no request follows the wait that ran out."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <set>
#include "qg_split_feed.h"

constexpr int STAGES = 7;

struct Ops {
  int fail_at, waits = 0;  // the wait that runs out (-1: none)
  bool failed = false, late = false, inputs = false;
  std::set<int> a, b;      // requested and not known to have landed
  bool wait() { return !(failed = waits++ == fail_at); }
  bool wait_a_free(int n) { if (!wait()) return false; a.erase(n - STAGES); return true; }
  bool wait_b_free(int u) { if (!wait()) return false; b.erase(u - 2); return true; }
  void wait_inputs() { inputs = true; }
  void load_a(int n, int, int) { late |= failed; a.insert(n); }
  void load_b(int u) { late |= failed || !inputs; b.insert(u); }
  void drain_a(int q) { a.erase(q); }
  void drain_b(int u) { b.erase(u); }
};

int main() {
  int runs = 0, bad = 0;
  for (int digits = 7; digits <= 8; ++digits)
    for (int units = 1; units <= 9; ++units)
      for (int f = -1;; ++f) {
        Ops o{f};
        qg::split_feed<STAGES>(o, units, digits);
        ++runs;
        if (o.late || !o.a.empty() || !o.b.empty()) {
          ++bad;
          std::printf("digits %d units %d wait %d: %zu of A, %zu of B in flight at the exit%s\n", digits, units, f, o.a.size(),
                      o.b.size(), o.late ? ", requests after the wait" : "");
        }
        if (f >= 0 && !o.failed) break;  // fewer waits than f
      }
  std::printf("%d runs, %d bad\n", runs, bad);
  return bad != 0 || runs < 100;
}
"""


def test_every_copy_requested_is_waited_for(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "feed.cpp", tmp_path / "feed"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2310_06650_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout[-2000:]
