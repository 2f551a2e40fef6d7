"""Buffers of an optional path (csrc/optional.h): with an allocator that fails at
the k-th request, none is kept, every pointer is null and a later try gets all
of them."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <set>
#include "optional.h"

int main() {
  int bad = 0;
  for (int fail = 0; fail <= 5; ++fail) {
    std::set<void*> held;
    int calls = 0;
    auto get = [&](size_t n) -> void* {
      if (calls++ == fail) return nullptr;
      void* q = std::malloc(n);
      held.insert(q);
      return q;
    };
    auto put = [&](void* q) {
      bad += held.erase(q) != 1;
      std::free(q);
    };
    int* a = (int*)1;
    double* b = (double*)1;
    char* c = (char*)1;
    auto ask = [&] { return vcsgc::get_all({vcsgc::wanted(&a, 3), vcsgc::wanted(&b, 0), vcsgc::wanted(&c, 7)}, get, put); };
    const bool ok = ask();
    bad += ok != (fail > 2);
    if (!ok) bad += a || b || c || !held.empty() || calls != fail + 1;
    else bad += !a || !b || !c || held.size() != 3;
    if (!ok) bad += !ask() || held.size() != 3;
  }
  std::printf("%d\n", bad);
  return bad;
}
"""


def test_all_or_none(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_1012_5082_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "0\n"
