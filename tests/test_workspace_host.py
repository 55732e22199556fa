"""A workspace whose allocation fails is made anew by the next call, whichever
of its buffers failed (the rule of workspace.h, compiled for the host with
buffers whose allocation throws at a chosen call)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1609_08130_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include "workspace.h"
static int calls = 0, fail_at = -1;
struct Buf {
  int size = 0;  // 0: no memory
  void alloc(int n) {
    size = 0;  // the old memory is released first
    if (calls++ == fail_at) throw 1;
    size = n;
  }
};
int main() {
  int bad = 0;
  for (int fail = 0; fail < 2; fail++) {
    Buf a, b;
    int have = 0, gen = 0;
    auto ensure = [&](int want) {
      rss::regrow(have, want, [&] { gen++; a.alloc(want); b.alloc(want); });
    };
    calls = 0, fail_at = -1;
    ensure(4);
    const int g0 = gen;
    ensure(4);
    ensure(1);
    bad += gen != g0 || calls != 2;  // nothing to do
    fail_at = calls + fail;
    bool threw = false;
    try {
      ensure(64);
    } catch (int) {
      threw = true;
    }
    bad += !threw || gen == g0;  // what captured the old buffers is told
    ensure(1);
    bad += a.size < 1 || b.size < 1 || have < 1;
    ensure(64);
    bad += a.size < 64 || b.size < 64 || have != 64;
  }
  printf("%d\n", bad);
  return 0;
}
"""


def test_failed_allocation_is_repeated(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "w.cpp", tmp_path / "w"
    src.write_text(SOURCE)
    subprocess.check_call([cxx, "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)])
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout
    assert out.split() == ["0"]
