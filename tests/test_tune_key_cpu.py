"""What the autotuner tells tilings and images apart by (csrc/tune_key.h, compiled for the host): an
image whose plan leaves the z-update to the library but whose weights rule out the pixel-domain
form runs the transform passes, so every field of theirs counts; and it does not share a tuned
tiling with an image of the other form."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_CODE = r"""
#include <cstdio>
#include "tune_key.h"
struct Row { int threads; };
struct Plan { int THmax, zl, QB, CB; Row row; int NSEG, zf_cs, rp, p2; };
static std::vector<int> key(const Plan& p, bool pixel) {
  std::vector<int> k;
  sgs::append_tiling_key(k, p, pixel);
  return k;
}
#define CHECK(x) if (!(x)) { std::printf("%s\n", #x); return 1; }
int main() {
  const Plan base{16, 1, 8, 8, {256}, 4, 0, 0, 0};
  Plan v[8] = {base, base, base, base, base, base, base, base};
  v[0].QB = 4; v[1].CB = 4; v[2].row.threads = 128; v[3].NSEG = 8;
  v[4].zf_cs = 2; v[5].rp = 1; v[6].p2 = 1;
  v[7].THmax = 8;
  for (int i = 0; i < 7; ++i) {
    CHECK(key(v[i], true) == key(base, true))      // the passes do not run
    CHECK(key(v[i], false) != key(base, false))    // larger weights: they do
    Plan a = v[i], b = base;
    a.zl = b.zl = 0;                               // the tiling asks for them
    CHECK(key(a, true) != key(b, true))
  }
  CHECK(key(v[7], true) != key(base, true) && key(v[7], false) != key(base, false))
  const sgs::TuneKey a = sgs::make_tune_key(0, 1, 8, 100, 120, true), b = sgs::make_tune_key(0, 1, 8, 100, 120, false),
                     c = sgs::make_tune_key(0, 1, 8, 128, 127, true), d = sgs::make_tune_key(0, 1, 8, 128, 128, true);
  CHECK((a < b) != (b < a))
  CHECK(!(a < c) && !(c < a) && c < d)
  return 0;
}
"""


def test_keys(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(_CODE)
    csrc = os.path.join(ROOT, "paper_1504_07028_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", csrc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
