"""How slots are dealt out to blocks (deal.h): every slot once, and in a factorised tick no
block with more candidates than warps while every candidate can have a warp."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1906_02318_gb300", "csrc")
PROGRAM = r"""
#include <stdio.h>
#include <vector>
#include "deal.h"
using namespace mpmi;
// n slots (listed: a device-side count below the launch's n) over the launch's blocks
static int check(int n, int listed, int sms) {
  int wpb, grid;
  fact_launch(n, sms, 32, &wpb, &grid);
  std::vector<char> seen(listed, 0);
  for (int b = 0; b < grid; ++b) {
    const FactShare in(listed, grid, wpb, b);
    if (b >= in.stride) continue;
    const int mine = in.count(listed);
    if (mine > wpb && listed <= grid * wpb) return printf("n %d of %d: block %d has %d for %d warps\n", listed, n, b, mine, wpb);
    if (listed >= in.stride && mine < 1) return printf("n %d of %d: block %d has none\n", listed, n, b);
    for (int i = 0; i < mine; ++i) {
      const int s = in.slot(i);
      if (s < 0 || s >= listed || seen[s]) return printf("n %d of %d: slot %d\n", listed, n, s);
      seen[s] = 1;
    }
  }
  for (int s = 0; s < listed; ++s)
    if (!seen[s]) return printf("n %d of %d: slot %d is left out\n", listed, n, s);
  return 0;
}
int main() {
  for (int n = 1; n <= 6000; ++n)
    if (check(n, n, 152)) return 1;
  const int sizes[] = {8191, 16384, 30001, 65536, 100003, 1048576};
  for (int n : sizes)
    for (int listed : {n, 1, 7, 31, 152, 700, 4863, 4865, n - 1})
      if (check(n, listed < n ? listed : n, 152)) return 1;
  for (int sms : {1, 2, 148})
    for (int n = 1; n <= 5000; n += 7)
      if (check(n, n, sms)) return 1;
  // sorted units: every slot once, no unit larger than the first
  for (int n : {1, 7, 8, 9, 62500, 65536, 1300001})
    for (int units : {1, 152, 304}) {
      std::vector<char> seen(n, 0);
      for (int u = 0; u < units; ++u)
        for (int i = 0; i < unit_count(n, units, u); ++i) {
          const int s = UnitSlots{u, units}.slot(i);
          if (unit_count(n, units, u) > unit_count(n, units, 0) || s >= n || seen[s]++)
            return printf("unit %d of %d over %d\n", u, units, n);
        }
      for (int s = 0; s < n; ++s)
        if (!seen[s]) return printf("slot %d of %d, %d units\n", s, n, units);
    }
  return 0;
}
"""


def test_slots_are_dealt_out_once_and_evenly(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    (tmp_path / "deal.cpp").write_text(PROGRAM)
    exe = tmp_path / "deal"
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", CSRC, str(tmp_path / "deal.cpp"), "-o",
                    str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
