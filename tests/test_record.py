"""The tagged record of a block's partial sums (cgp_fixed.h: pack_record) on the CPU: every field comes
back, and a record reads as current for its own reduction only."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_00082_gb300", "csrc")

SOURCE = r"""
#include <random>
#include "cgp_fixed.h"
using namespace cgp::fx;
int main() {
  std::mt19937_64 rng(5);
  const int64_t top = (1ll << 62) - 1;
  for (int i = 0; i < 200000; ++i) {
    int64_t S[3];
    int E[3];
    uint64_t w[4];
    for (int c = 0; c < 3; ++c) {
      S[c] = i < 8 ? ((i >> c) & 1 ? top : -top) : (int64_t)rng() >> (2 + rng() % 62);
      E[c] = i < 8 ? (i & 1 ? 1 : 2046) : 1 + (int)(rng() % 2046);
    }
    if (i % 5 == 0) E[i % 3] = kBadExp;
    const int red = (int)(rng() % 1000000);
    pack_record(S, E, red, w);
    for (int other = red - 6; other <= red + 6; ++other)
      if (other >= 0 && record_current(w, record_tag(other)) != (other == red)) return 1;
    for (int c = 0; c < 3; ++c) {
      if (record_exponent(w, c) != E[c]) return 2;
      if (record_mantissa(w, c) != (E[c] == kBadExp ? 0 : S[c])) return 3;
    }
    uint64_t v[4];   // any one word from another reduction
    for (int c = 0; c < 4; ++c) v[c] = w[c];
    v[i % 4] = (v[i % 4] & ~0xFFull) | record_tag(red + 2);
    if (record_current(v, record_tag(red))) return 4;
  }
  const uint64_t none[4] = {0, 0, 0, 0};
  for (int red = 0; red < 600; ++red)
    if (record_current(none, record_tag(red))) return 5;
  return 0;
}
"""


def test_record_round_trip_and_tags(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src = tmp_path / "record.cpp"
    src.write_text(SOURCE)
    exe = str(tmp_path / "record")
    subprocess.run([gxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
