// Chains of coordinates that share a bucket: the arithmetic behind the chained insert.
//
// For c a power of two the bucket of coordinate i is a rotation.  p = 2^61 - 1 is -1 modulo c, so
// adding a to a hash value x and subtracting p on a wrap moves the bucket x mod c by a mod c, plus
// one on a wrap: with pos(i) = (x mod c) + x/p on the circle of length c,
//   pos(i + S) = pos(i) + S * theta (mod c),   theta = (a mod c) + a/p,   bucket = floor(pos).
// A stride S for which S * theta is close to a multiple of c therefore keeps a coordinate's
// bucket: of the coordinates i, i + S, i + 2S, ... consecutive ones lie in the same bucket except
// once in 1/|delta| steps, delta = S * theta mod c taken in (-c/2, c/2].  Such strides exist for
// every theta: the convergents q_n of theta/c satisfy |delta(q_n)| < c / q_{n+1}.
//
// Everything here only chooses strides; a poor choice costs time, never a result.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

namespace gs {

// One convergent (or small start value) of a row's rotation: stride q and its drift in buckets.
struct Convergent {
  int64_t q;
  double delta;
};

// The convergents of theta/c with denominators below 2^31, from a Euclidean expansion of
// ((a mod c) * p + a) / (c * p).
inline std::vector<Convergent> rotation_convergents(uint64_t a, uint32_t c) {
  typedef unsigned __int128 u128;
  const u128 p = ((u128)1 << 61) - 1;
  const u128 den = p * c;
  const u128 num = ((u128)(a % c)) * p + a;  // < den
  // q_n num is a multiple of den plus (-1)^n times the n-th remainder of the expansion
  std::vector<Convergent> out;
  u128 x = den, y = num;
  int64_t q0 = 0, q1 = 1;  // denominators of the last two convergents
  double sign = 1.0;
  out.push_back({1, (double)y / (double)p});
  while (y != 0) {
    const u128 k = x / y;
    const u128 next = k * (u128)q1 + (u128)q0;
    if (next >= ((u128)1 << 31)) break;
    const u128 t = x - k * y;
    x = y;
    y = t;
    q0 = q1;
    q1 = (int64_t)next;
    sign = -sign;
    const Convergent v = {q1, sign * ((double)y / (double)p)};
    if (q1 > out.back().q) out.push_back(v);
    else out.back() = v;
  }
  return out;
}

// How a row's coordinates are walked: chains of `steps` coordinates `stride` apart.
struct ChainShape {
  int64_t stride;
  int32_t steps;
  double flushes;  // expected cell updates per coordinate
};

// The stride and chain length with the fewest cell updates per coordinate,
// min(1, |delta(S)|) + 1/steps, with stride >= min_stride and steps <= max_steps.
// Candidates are the smallest usable multiples of the convergents and the sums k q_n + q_{n-1}.
inline ChainShape choose_chain(const std::vector<Convergent>& cv, int64_t d, int64_t min_stride, int64_t max_steps) {
  ChainShape best = {d, 1, 1.0};
  const auto consider = [&](int64_t S, double delta) {
    if (S < min_stride || S >= d) return;
    int64_t steps = (d + S - 1) / S;
    if (steps > max_steps) steps = max_steps;
    const double drift = std::fabs(delta) < 1.0 ? std::fabs(delta) : 1.0;
    double f = drift + 1.0 / (double)steps;
    const double full = (double)d / (double)S;  // a last, partly filled step counts as what it covers
    if (full < (double)steps) f = drift + 1.0 / full;
    if (f < best.flushes) best = {S, (int32_t)steps, f};
  };
  for (size_t n = 0; n < cv.size(); ++n) {
    const int64_t q = cv[n].q;
    const int64_t k0 = q >= min_stride ? 1 : (min_stride + q - 1) / q;
    consider(k0 * q, (double)k0 * cv[n].delta);
    consider((k0 + 1) * q, (double)(k0 + 1) * cv[n].delta);
    if (n == 0) continue;
    const int64_t q0 = cv[n - 1].q;
    const int64_t a = n + 1 < cv.size() ? (cv[n + 1].q - q0) / q : (((int64_t)1 << 31) - q0) / q;
    int64_t k1 = q0 >= min_stride ? 1 : (min_stride - q0 + q - 1) / q;
    if (k1 < 1) k1 = 1;
    if (k1 <= a) consider(k1 * q + q0, (double)k1 * cv[n].delta + cv[n - 1].delta);
  }
  return best;
}

// Strides with |drift| < 1/2 that are small combinations k q_n + l q_{n-1} of two neighbouring
// convergents, ascending.
inline std::vector<Convergent> slow_strides(const std::vector<Convergent>& cv, int64_t min_stride) {
  std::vector<Convergent> out;
  for (size_t n = 0; n < cv.size(); ++n)
    for (int64_t k = 1; k <= 4; ++k)
      for (int64_t l = 0; l <= (n > 0 ? 2 : 0); ++l) {
        const int64_t q = k * cv[n].q + (l ? l * cv[n - 1].q : 0);
        const double delta = (double)k * cv[n].delta + (l ? (double)l * cv[n - 1].delta : 0.0);
        if (q >= min_stride && q < ((int64_t)1 << 31) && std::fabs(delta) < 0.5) out.push_back({q, delta});
      }
  std::sort(out.begin(), out.end(), [](const Convergent& x, const Convergent& y) { return x.q < y.q; });
  return out;
}

// A walk that serves two rows: i = base + m * inner + n * outer with base < inner, base + m * inner < outer,
// m < inner_steps and n < outer_steps, and the same again from every multiple of outer * outer_steps.
// Along m the first row keeps its buckets, along n the second.
struct PairShape {
  int64_t inner = 0, outer = 0;
  int32_t inner_steps = 0, outer_steps = 0;
  double changes = 2.0;  // expected bucket changes per coordinate, both rows
};

// Both lists ascending.  An inner stride serves an outer one only from outer / max_inner on, so the
// search starts there, and a pair is given up before its divisions once a bound from below on its
// bucket changes reaches the best found (the factor covers the bound's own rounding).  Every direct
// query along a walk pays for two of these searches on the host, about 80 x 80 pairs each: 3 to 8 us
// for both, 20 to 43 when every pair is evaluated (c = 2^16 to 2^21).
inline PairShape choose_pair(const std::vector<Convergent>& first, const std::vector<Convergent>& second, int64_t d,
                             int max_inner, int64_t max_steps) {
  PairShape best;
  size_t from = 0;
  for (const Convergent& o : second) {
    if (o.q >= d) break;
    while (from < first.size() && first[from].q * max_inner < o.q) ++from;
    const double inverse = 1.0 / (double)o.q;
    // a round has two inner steps or more, so the walk at most max_steps / 2 rounds
    const double rest = std::fabs(o.delta) + std::max((double)o.q / (double)d, 2.0 / (double)max_steps);
    if ((rest + 1.0 / max_inner) * (1.0 - 1e-9) >= best.changes) continue;
    for (size_t at = from; at < first.size(); ++at) {
      const Convergent& s = first[at];
      if (s.q >= o.q) break;
      if ((std::fabs(s.delta) + (double)s.q * inverse + rest) * (1.0 - 1e-9) >= best.changes) continue;
      const int64_t m = (o.q + s.q - 1) / s.q;
      int64_t n = (d + o.q - 1) / o.q;
      if (n * m > max_steps) n = max_steps / m;
      if (n < 1) continue;
      const double reach = std::min((double)n, (double)d / (double)o.q);
      const double changes = std::fabs(s.delta) + (double)s.q / (double)o.q + std::fabs(o.delta) + 1.0 / reach;
      if (changes < best.changes) best = {s.q, o.q, (int32_t)m, (int32_t)n, changes};
    }
  }
  return best;
}

inline uint64_t mulmod61(uint64_t a, uint64_t b) {
  const unsigned __int128 p = ((unsigned __int128)1 << 61) - 1;
  return (uint64_t)((unsigned __int128)a * b % p);
}

}  // namespace gs
