"""Host checks of the chained insert's strides (csrc/chain_plan.h), compiled with the host compiler:
the drift of every convergent against buckets evaluated from the hash's definition, and the walk over
segments, chains and steps, which has to visit every coordinate exactly once for any length."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_06004_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "chain_plan.h"
using namespace gs;
static const uint64_t P = (1ull << 61) - 1;
static uint64_t hash(uint64_t a, uint64_t b, int64_t i) { return (uint64_t)(((unsigned __int128)a * i + b) % P); }
int main() {
  const uint64_t as[] = {1, 2, P - 1, P - 2, 0x123456789ABCDEFull, 987654321987654321ull, (1ull << 60) + 12345, 1ull << 43};
  const uint32_t cs[] = {1, 2, 64, 1u << 14, 1u << 21, 1u << 26};
  const int64_t ds[] = {1, 2, 255, 256, 257, 4095, 4096, 4097, 8193, 100003, 1234567};
  for (uint64_t a : as)
    for (uint32_t c : cs) {
      const auto cv = rotation_convergents(a, c);
      for (const Convergent& v : cv) {
        if (v.q < 1 || v.q >= (1ll << 31) || std::fabs(v.delta) > 0.5 * c + 1e-6) return 1;
        for (int64_t i = 0; i < 200; ++i) {  // the bucket moves by floor(delta) or floor(delta) + 1
          const uint64_t b = 0x1234567ull;
          const int64_t m = (int64_t)(hash(a, b, i + v.q) % c) - (int64_t)(hash(a, b, i) % c);
          const int64_t lo = (int64_t)std::floor(v.delta - 1e-9), hi = (int64_t)std::floor(v.delta + 1e-9) + 1;
          bool ok = false;
          for (int64_t k = lo; k <= hi; ++k) ok = ok || (m - k) % (int64_t)c == 0;
          if (!ok) return 2;
        }
      }
      for (int64_t d : ds)
        for (int64_t max_steps : {1, 5, 32}) {
          const ChainShape ch = choose_chain(cv, d, 4096, max_steps);
          if (ch.stride < 1 || ch.steps < 1 || ch.steps > max_steps) return 3;
          std::vector<char> seen((size_t)d, 0);
          const int64_t span = ch.stride * ch.steps;
          for (int64_t seg = 0; seg < (d + span - 1) / span; ++seg)
            for (int64_t t = 0; t < ch.stride; ++t)
              for (int64_t n = 0, i = seg * span + t; n < ch.steps && i < d; ++n, i += ch.stride)
                if (seen[(size_t)i]++) return 4;
          for (char s : seen)
            if (!s) return 5;
        }
    }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_chain_plan(tmp_path):
    src = tmp_path / "check.cpp"
    src.write_text(MAIN)
    exe = tmp_path / "check"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
