"""The lifting's feature codes (basis.h) against feature_split, every basis and feature,
bit for bit in float32 (the codes take the same products in the same order)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1906_02318_gb300", "csrc")
PROGRAM = r"""
#include <stdio.h>
#include <string.h>
#include "basis.h"
using namespace mpmi;
int main() {
  const float x[6] = {0.3f, -1.7f, 2.9f, 13.1f, -0.07f, 0.41f};
  const float s = 0.6234f, c = -0.7819f;
  float v[16] = {1.f};
  for (int i = 0; i < 6; ++i) v[kVX + i] = x[i];
  v[kVSin] = s;
  v[kVCos] = c;
  int checked = 0;
  for (int kind = kBot; kind <= kLin41; ++kind) {
    int n, nx, nu, np;
    kind_dims(kind, &n, &nx, &nu, &np);
    for (int j = 0; j < n; ++j) {
      float a, b[kMaxP], wa, wb[kMaxP];
      feature_split<float>(kind, j, x, s, c, &wa, wb);
      const uint32_t f = feature_code(kind, j);
      a = v[f & 15] * v[f >> 4 & 15] * v[f >> 8 & 15];
      for (int k = 0; k < kMaxP; ++k) b[k] = (f >> 16) == (uint32_t)k ? v[f >> 12 & 15] : 0.f;
      if (memcmp(&a, &wa, 4) || memcmp(b, wb, sizeof b)) {
        printf("basis %d feature %d\n", kind, j);
        return 1;
      }
      ++checked;
    }
  }
  return checked == 12 + 32 + 2 + 4 + 5 ? 0 : 2;
}
"""


def test_feature_codes_equal_feature_split(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    (tmp_path / "codes.cpp").write_text(PROGRAM)
    exe = tmp_path / "codes"
    subprocess.run([gxx, "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC,
                    str(tmp_path / "codes.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
