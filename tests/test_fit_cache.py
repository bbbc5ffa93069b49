"""The remembered occupancy answers of the selection kernel (plain C++)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include "fit_cache.h"
using namespace stl;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
static FitCache<2, 16, 4> cache;
int main() {
  // an answer counts in the context it was given in, and there only
  CHECK(cache.get(0, 8, 2, 7) == -1);
  cache.put(0, 8, 2, 7, 3);
  CHECK(cache.get(0, 8, 2, 7) == 3);
  CHECK(cache.get(0, 8, 2, 9) == -1);
  CHECK(cache.get(1, 8, 2, 7) == -1 && cache.get(0, 7, 2, 7) == -1 && cache.get(0, 8, 1, 7) == -1);
  cache.put(0, 8, 2, 9, 19);
  CHECK(cache.get(0, 8, 2, 9) == 19 && cache.get(0, 8, 2, 7) == -1);
  // "none fit" in a small context takes the size from nobody
  cache.put(0, 16, 1, 7, 0);
  CHECK(cache.get(0, 16, 1, 7) == -1);
  // no context, or a device past the table: always asked
  cache.put(0, 4, 1, 0, 5);
  CHECK(cache.get(0, 4, 1, 0) == -1);
  cache.put(2, 4, 1, 7, 5);
  CHECK(cache.get(2, 4, 1, 7) == -1);
  // the size asked for covers every size it answers for
  const int sm = 233472, fixed = 1024 + 13660, most = 4, cap = 49152 * 4;
  for (int dyn = 16; dyn <= cap; dyn += 16) {
    const int occ = ctas_per_sm(sm, fixed, dyn, most);
    CHECK(occ >= 1);
    const int big = largest_dynamic(sm, fixed, occ, cap);
    CHECK(big >= dyn && big % 16 == 0 && big <= cap && ctas_per_sm(sm, fixed, big, most) == occ);
  }
  std::puts("ok");
  return 0;
}
"""


def test_fit_cache(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2603_00188_gb300", "csrc"),
                    str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "ok\n"
