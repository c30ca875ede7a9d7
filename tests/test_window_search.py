"""The window searches' index arithmetic, compiled for the host from the
kernels' own header: every search finds the first entry of weight >= t and
reads no entry outside its row, also where the row ends at the largest
accepted adjacency (2m = 2^32 - 2)."""
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2506_19349_gb300" / "csrc"

PROGRAM = r"""
#include <stdio.h>
#include <initializer_list>

#include "search.h"

struct Row {  // entries [p, e): `light` of weight 1, then weight 9
  uint32_t p, e, light;
  bool* out;
  uint32_t operator()(uint32_t i) const {
    if (i < p || i >= e) *out = true;
    return i - p < light ? 1u : 9u;
  }
};

int main() {
  const uint32_t ends[] = {100u, 0x7FFFFFFFu, 0x80000001u, 0xFFFFFFF0u, 0xFFFFFFFEu};
  for (uint32_t e : ends)
    for (uint32_t len = 0; len <= 40; ++len)
      for (uint32_t light = 0; light <= len; ++light)
        for (int64_t t : {1ll, 2ll, 9ll, 10ll, 1ll << 33}) {
          bool out = false;
          const Row w = {e - len, e, light, &out};
          const uint32_t b = e - len, want = t <= 1 ? b : t <= 9 ? b + light : e;
          const uint32_t got[] = {eic::lower_bound(w, b, e, t), eic::gallop(w, b, e, t), eic::gallop4(w, b, e, t)};
          for (int k = 0; k < 3; ++k)
            if (got[k] != want || out) {
              printf("search %d: row [%u, %u), %u light, t %lld: %u, not %u%s\n", k, b, e, light, (long long)t, got[k], want,
                     out ? "; an entry outside the row was read" : "");
              return 1;
            }
        }
  return 0;
}
"""


def test_window_searches(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "search.cpp", tmp_path / "search"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-I", str(CSRC), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
