"""The bounded map that keeps a group's captured iterations: keys cycled through
within its bound are all found again, and a full one gives up the least
recently used object alone."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <set>
#include "henry_recent.cuh"
int main() {
  typedef hk::RecentMap<int, int, 256> Map;
  std::multiset<int> gone;
  auto drop = [&](int v) { gone.insert(v); };
  for (int sizes : {1, 16, 17, 41, 256}) {  // two rounds: the second one builds nothing
    Map m;
    int built = 0;
    for (int round = 0; round < 2; ++round)
      for (int k = 0; k < sizes; ++k)
        if (int* v = m.find(k)) {
          if (*v != 10 * k) return 1;
        } else {
          if (*m.insert(k, 10 * k, drop) != 10 * k) return 2;
          ++built;
        }
    if (built != sizes || !gone.empty() || (int)m.size() != sizes) return 3;
  }
  Map m;
  for (int k = 0; k < 256; ++k) m.insert(k, k, drop);
  for (int k = 0; k < 256; k += 2) m.find(k);  // the odd ones are now the oldest
  for (int k = 0; k < 128; ++k) m.insert(1000 + k, 1000 + k, drop);
  if (m.size() != 256 || gone.size() != 128) return 4;
  for (int k = 0; k < 256; ++k)
    if ((m.find(k) != nullptr) != (k % 2 == 0) || (gone.count(k) == 1) != (k % 2 == 1)) return 5;
  Map copy = m;  // values move with the group that owns them
  if (!copy.find(0) || !copy.find(1127)) return 6;
  gone.clear();
  m.clear(drop);
  if (m.size() != 0 || gone.size() != 256 || m.find(0)) return 7;
  m.insert(5, 6, drop);
  return m.find(5) && *m.find(5) == 6 ? 0 : 8;
}
"""


def test_recent_map(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "recent.cpp", tmp_path / "recent"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", os.path.join(ROOT, "paper_2302_07804_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
