"""The bookkeeping by which the warps of a path-A level reserve cache ids, run
on the CPU (the header that the kernel uses, compiled as plain C++): every claim
gets an id of its own, no reserved id is lost, and what a warp leaves over is one
range of at most kLanesAhead ids, however many of its claims are lost to others."""
from __future__ import annotations

import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <random>
#include <vector>
#include "lsyn_ids.h"
using namespace lsyn;

int main(int argc, char** argv) {
  const int warps = std::atoi(argv[1]), rounds = std::atoi(argv[2]);
  const unsigned ahead = unsigned(std::atoi(argv[3])), most = unsigned(std::atoi(argv[4]));
  std::mt19937 rng(7);
  unsigned counter = 0;
  std::vector<IdStock> stock(warps);
  std::vector<char> used;
  for (int i = 0; i < rounds; ++i)
    for (auto& s : stock) {
      const unsigned empty = rng() % (most + 1), n = empty ? rng() % (empty + 1) : 0u;  // some claims are lost
      const unsigned left = unsigned(rounds - 1 - i);
      const unsigned asked = n ? s.ask(n, ahead < 2 * left ? ahead : 2 * left) : 0u, fresh = counter;
      counter += asked;
      used.resize(counter, 0);
      for (unsigned r = 0; r < n; ++r) {
        const unsigned id = s.id(r, fresh);
        if (id >= counter || used[id]) return std::printf("id %u given twice or never reserved\n", id), 1;
        used[id] = 1;
      }
      if (n) s.use(n, asked, fresh);
    }
  unsigned long long over = 0, unused = 0;
  for (auto& s : stock) {
    if (s.end < s.next || s.have() > ahead) return std::printf("a warp leaves %u over\n", s.have()), 1;
    for (unsigned id = s.next; id < s.end; ++id)
      if (used[id]) return std::printf("id %u is in a stock and used\n", id), 1;
    over += s.have();
  }
  for (char u : used) unused += !u;
  if (unused != over) return std::printf("%llu ids unused, %llu in stocks\n", unused, over), 1;
  std::printf("%u %llu\n", counter, over);
  return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("ids")
    (d / "ids.cpp").write_text("#include <cstdlib>\n" + PROGRAM)
    csrc = os.path.join(ROOT, "paper_2504_18943_gb300", "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", csrc, "-o", str(d / "ids"), str(d / "ids.cpp")], check=True)
    return str(d / "ids")


@pytest.mark.parametrize("ahead", [0, 1, 64])
@pytest.mark.parametrize("most", [1, 32, 128])  # empty slots that a warp batch meets at most
def test_no_id_is_lost(program, ahead, most):
    for rounds in (1, 2, 500):
        r = subprocess.run([program, "40", str(rounds), str(ahead), str(most)], capture_output=True, text=True)
        assert r.returncode == 0, r.stdout
