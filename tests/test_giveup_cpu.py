"""The exit after an exhausted wait (csrc/giveup.h, compiled for the host): in every interleaving of
a few threads and rows, with one barrier a row, whichever threads give up in whichever rows, all
threads of a sweep CTA leave after the same row; and the wait for copies in flight is a
millisecond at the clock of the GPU (2.07 GHz) however short the budget."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_CODE = r"""
#include <cstdio>
#include <set>
#include <tuple>
#include <vector>
#include "giveup.h"
constexpr int NT = 3, ROWS = 4;
// a thread's next action in its row: 0 wait (raise the flag if it gives up), 1 at the barrier,
// 2 read the flag; left: the row after which it returned (-1: none)
struct Thread { int row, step, left; };
struct State {
  int flag[2];
  Thread t[NT];
  bool operator<(const State& o) const { return key() < o.key(); }
  std::vector<int> key() const {
    std::vector<int> k{flag[0], flag[1]};
    for (auto& x : t) { k.push_back(x.row); k.push_back(x.step); k.push_back(x.left); }
    return k;
  }
};
static unsigned quits;                 // bit row * NT + thread: that wait runs out
static std::set<State> seen;
static bool parted;
static void walk(State s) {
  if (!seen.insert(s).second) return;
  bool done = true;
  for (int i = 0; i < NT; ++i) {
    State n = s;
    Thread& x = n.t[i];
    if (x.left >= 0 || x.row == ROWS) continue;
    done = false;
    const sgs::GiveUp g{n.flag};
    if (x.step == 0) {
      if (quits >> (x.row * NT + i) & 1) g.raise(x.row);
      x.step = 1;
    } else if (x.step == 1) {          // passes when every thread that has not left is at this barrier
      for (int j = 0; j < NT; ++j)
        if (s.t[j].left < 0 && (s.t[j].row != x.row || s.t[j].step < 1)) goto next;
      for (int j = 0; j < NT; ++j)
        if (n.t[j].left < 0) n.t[j].step = 2;
    } else if (g.raised(x.row)) {
      x.left = x.row;
    } else {
      ++x.row;
      x.step = 0;
    }
    walk(n);
  next:;
  }
  if (done)
    for (int i = 1; i < NT; ++i) parted |= s.t[i].left != s.t[0].left;
}
int main() {
  for (long long b : {1LL, 200000LL, 2000000000LL})
    if (sgs::drain_cycles(b) < b || sgs::drain_cycles(b) < 2070000LL) { std::printf("drain %lld\n", b); return 1; }
  for (quits = 0; quits < 1u << (NT * ROWS); ++quits) {
    State s{};
    for (auto& x : s.t) x.left = -1;
    sgs::GiveUp{s.flag}.clear();
    seen.clear();
    walk(s);
    if (parted) { std::printf("threads part for %x\n", quits); return 1; }
    if (quits)                         // somebody gave up: nobody stays
      for (auto& e : seen)
        for (auto& x : e.t)
          if (x.row == ROWS) { std::printf("a thread stays for %x\n", quits); return 1; }
  }
  return 0;
}
"""


def test_threads_leave_together(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(_CODE)
    csrc = os.path.join(ROOT, "paper_1504_07028_gb300", "csrc")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", csrc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
