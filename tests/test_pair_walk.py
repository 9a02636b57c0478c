"""Host checks of the walk that serves two rows (choose_pair in csrc/chain_plan.h), compiled with the host
compiler: the choice against a search of every pair, at a fraction of its time; the walk of the query
kernel, restated, visits every coordinate once, stays within the inner steps it may take, and ends each
round at the last inner step or the one before, for which the jumps to the next round exist."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2108_06004_gb300", "csrc")

MAIN = r"""
#include <chrono>
#include <cstdio>
#include <cstring>
#include <random>
#include "chain_plan.h"
using namespace gs;
typedef std::vector<Convergent> List;

static PairShape search_all(const List& first, const List& second, int64_t d, int max_inner, int64_t max_steps) {
  PairShape best;
  for (const Convergent& o : second)
    for (const Convergent& s : first) {
      if (o.q >= d || s.q >= o.q) continue;
      const int64_t m = (o.q + s.q - 1) / s.q;
      int64_t n = (d + o.q - 1) / o.q;
      if (n * m > max_steps) n = max_steps / m;
      if (m > max_inner || n < 1) continue;
      const double reach = std::min((double)n, (double)d / (double)o.q);
      const double changes = std::fabs(s.delta) + (double)s.q / (double)o.q + std::fabs(o.delta) + 1.0 / reach;
      if (changes < best.changes) best = {s.q, o.q, (int32_t)m, (int32_t)n, changes};
    }
  return best;
}

static bool walk(const PairShape& w, int64_t d, std::vector<char>& seen) {
  const uint32_t S0 = (uint32_t)w.inner, S1 = (uint32_t)w.outer, D = (uint32_t)d;
  const int64_t span = w.outer * w.outer_steps;
  seen.assign((size_t)d, 0);
  for (int64_t seg = 0; seg < (d + span - 1) / span; ++seg)
    for (uint32_t base = 0; base < S0; ++base) {
      if (seg * span + base >= d) break;
      uint32_t i = (uint32_t)(seg * span + base), round = i;
      int m = 0, n = 0;
      for (bool live = true; live;) {
        if (m >= w.inner_steps || i >= D || seen[i]++) return false;
        if (i - round + base + S0 < S1 && i + S0 < D) {
          i += S0;
          ++m;
          continue;
        }
        const int at = m;
        i = round + S1;
        round = i;
        m = 0;
        ++n;
        live = n < w.outer_steps && i < D;
        if (live && at != w.inner_steps - 1 && at != w.inner_steps - 2) return false;
      }
    }
  return std::memchr(seen.data(), 0, (size_t)d) == nullptr;
}

int main() {
  std::mt19937_64 rng(11);
  const uint64_t P = (1ull << 61) - 1;
  std::vector<char> seen;
  double fast = 0, slow = 0;
  int served = 0;
  for (uint32_t c : {1u << 16, 1u << 18, 1u << 20, 1u << 21})
    for (int64_t d : {(int64_t)1 << 22, (int64_t)6000003, (int64_t)25557032, (int64_t)138357544, ((int64_t)1 << 31) - 1})
      for (int t = 0; t < 8; ++t) {
        List l[2];
        for (List& x : l) x = slow_strides(rotation_convergents(rng() % (P - 1) + 1, c), 4096);
        const int64_t max_steps = std::min<int64_t>(64, d / (152 * 2048));
        const auto t0 = std::chrono::steady_clock::now();
        const PairShape a = choose_pair(l[0], l[1], d, 8, max_steps);
        const auto t1 = std::chrono::steady_clock::now();
        const PairShape b = search_all(l[0], l[1], d, 8, max_steps);
        const auto t2 = std::chrono::steady_clock::now();
        fast += std::chrono::duration<double>(t1 - t0).count();
        slow += std::chrono::duration<double>(t2 - t1).count();
        if (a.inner != b.inner || a.outer != b.outer || a.inner_steps != b.inner_steps ||
            a.outer_steps != b.outer_steps || a.changes != b.changes) return 1;
        if (a.changes > 1.0) continue;
        ++served;
        if (a.inner < 4096 || a.inner_steps < 2 || a.inner_steps > 8) return 2;
        if (a.inner * (a.inner_steps - 1) >= a.outer) return 3;  // both jumps to a next round are forward
        if (d < (1 << 25) && t < 3 && !walk(a, d, seen)) return 4;
      }
  std::printf("%d pairs, %.0f us against %.0f us\n", served, fast * 1e6, slow * 1e6);
  return served < 40 ? 5 : fast * 5 > slow ? 6 : 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_pair_walk(tmp_path):
    src = tmp_path / "check.cpp"
    src.write_text(MAIN)
    exe = tmp_path / "check"
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, f"check {res.returncode} failed: {res.stdout}"
