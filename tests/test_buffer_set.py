"""The context's buffers grow in sets, all or none (csrc/bufferset.h): a C++ program puts in an allocator
that fails at each place in turn. After a failure no pointer is left (nothing dangling, nothing half
made) and nothing leaks; the next growth makes the whole set."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1501_01855_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include <stdlib.h>
#include <set>
#include "bufferset.h"
static std::set<void*> live;
static int calls, fail_at;
static int take(void** p, size_t n) {
  if (calls++ == fail_at) return 2;          // the pointer keeps what it held
  *p = malloc(n);
  live.insert(*p);
  return 0;
}
static void give(void* p) {
  if (live.erase(p) != 1) { printf("released twice\n"); exit(1); }
  free(p);
}
int main() {
  for (int k = 0; k < 3; ++k) {
    void *a = nullptr, *b = nullptr, *c = nullptr;
    fail_at = -1;
    if (ovl::renew_all({{&a, 8}, {&b, 16}, {&c, 24}}, take, give) != 0 || live.size() != 3) return 2;
    calls = 0;
    fail_at = k;
    if (ovl::renew_all({{&a, 80}, {&b, 160}, {&c, 240}}, take, give) != 2) return 3;
    if (a || b || c || !live.empty()) return 4;
    fail_at = -1;
    if (ovl::renew_all({{&a, 80}, {&b, 160}, {&c, 240}}, take, give) != 0 || !a || !b || !c) return 5;
    for (void* p : {a, b, c}) give(p);
  }
  return live.empty() ? 0 : 6;
}
"""


def test_a_failed_growth_leaves_nothing(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "set.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "set")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, (r.returncode, r.stdout)
