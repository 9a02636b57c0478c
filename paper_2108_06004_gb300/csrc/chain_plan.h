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
  std::vector<Convergent> out;
  u128 x = den, y = num;
  int64_t q0 = 0, q1 = 1;  // denominators of the last two convergents
  const auto drift = [&](int64_t q) {
    const u128 s = (u128)q * num % den;      // < 2^31 * 2^87
    return s <= den / 2 ? (double)s / (double)p : -((double)(den - s) / (double)p);
  };
  out.push_back({1, drift(1)});
  while (y != 0) {
    const u128 k = x / y;
    const u128 next = k * (u128)q1 + (u128)q0;
    if (next >= ((u128)1 << 31)) break;
    const u128 t = x % y;
    x = y;
    y = t;
    q0 = q1;
    q1 = (int64_t)next;
    if (q1 > out.back().q) out.push_back({q1, drift(q1)});
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

inline uint64_t mulmod61(uint64_t a, uint64_t b) {
  const unsigned __int128 p = ((unsigned __int128)1 << 61) - 1;
  return (uint64_t)((unsigned __int128)a * b % p);
}

}  // namespace gs
