"""The last pulls of a standalone commit + pull call (csrc/last_pulls.h),
compiled alone with the host compiler: the pulls that write are each worker's
last one, the counts agree, without a table every pull writes, and none of it
takes memory from the heap (agn_commit_pull_noalloc promises that)."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1710_02368_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#include <new>
#include "last_pulls.h"
static long g_news = 0;
void* operator new(std::size_t n) { ++g_news; void* p = std::malloc(n); if (!p) throw std::bad_alloc(); return p; }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
static int32_t table[agn::kStackPullWorkers], pw[600];
int main() {
  unsigned x = 12345;
  for (int n : {1, 2, 7, 64, agn::kStackPullWorkers}) {
    for (int R : {0, 1, 5, 600}) {
      for (int p = 0; p < R; ++p) pw[p] = (x = x * 1664525u + 1013904223u) / 65536 % n;
      const agn::LastPulls last(pw, R, table), every(pw, R, nullptr);
      for (int a = 0; a <= R; a += 3) {
        int k = 0;
        for (int p = a; p < R; ++p) {
          bool later = false;
          for (int q = p + 1; q < R; ++q) later |= pw[q] == pw[p];
          if (last.writes(p) == later || !every.writes(p)) return 1;
          k += !later;
        }
        if (last.count(a, R) != k || every.count(a, R) != R - a) return 2;
      }
    }
  }
  std::printf("%ld\n", g_news);
  return 0;
}
"""


def test_each_workers_last_pull_without_the_heap(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "last_pulls.cpp", tmp_path / "last_pulls"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.returncode
    assert out.stdout.strip() == "0"

