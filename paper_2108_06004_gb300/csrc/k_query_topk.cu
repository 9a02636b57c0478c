// Steps 4 and 5: median-of-r query of the merged sketch and top-k selection
// (Alg. 2 steps 1-3, read as a deterministic top-k by |est| with ties to the smaller index).
//
// The selection is a radix select on a 32-bit key in three levels: bits 31..21, 20..10 and
// 9..0.  For the top-k by |est| the key is the bit pattern of |est| (for non-negative floats
// it orders like the value); HEAVYMIX selects on a composite key (see heavy_key).  Each
// histogram kernel ends with a pick: the last CTA to finish (found with a counter after a
// memory fence, so no CTA waits for another) finds the bin that holds the k-th largest key
// and how many keys of that bin are still to be taken.  After three levels the k-th largest
// key tau is exact, and need_eq = k - #{key > tau} keys equal to tau are taken, those of
// smallest index.  Output indices are ascending.
//
// With a caller workspace (gs_query_topk):
//   k_qsample     (only where rows are pruned) the full estimate of a fixed strided sample of
//                 coordinates, its level-1 histogram, and a prune key from it: a lower bound
//                 on the k-th largest |est| of this query, rounded down to a bin edge
//   k_query       est_i for every i (fp32) + level-1 histogram + pick; when the estimate stays
//                 in the workspace, a coordinate whose rows read so far bound its |est| below
//                 the prune key skips its other rows and stores a marker (see below).  In its place:
//                 k_query_bits (pruning, the first rows' cells classified in shared memory),
//                 k_query_walk (long vectors, along a walk that keeps two rows' cells) and
//                 k_query_mod (c not a power of two); k_query_quads (HEAVYMIX: k_query) behind k_query_bits
//                 takes the query over where few coordinates settle early
//   k_repair      runs only if the level-1 pick fell below the prune key: recomputes every
//                 marked estimate in full, rebuilds the level-1 histogram and picks again
//   k_cand        one pass over est: keys above the picked level-1 bin are selected for
//                 certain and set their bit in a d-bit bitmap; keys inside the bin become
//                 candidates (index, key) and feed the level-2 histogram + pick
//   k_cand_hist3  level-3 histogram of the candidates + pick
//   k_cand_mark   candidates above tau into the bitmap, candidates equal to tau into a second
//   k_bm_count    per block of 65536 coordinates: bits set in each bitmap
//   k_scan        one CTA: exclusive prefix sums over the blocks
//   k_bm_write    every block writes its selected indices at their final positions
// Up to d = 1.5 * 2^20 (large k: 819,200) one launch of k_select_small replaces k_cand .. k_bm_write, where
// the device can hold its cluster.
// With the fixed scratch (gs_query_topk_noalloc), which cannot hold candidate lists, the
// levels 2 and 3 and the final selection read est in full passes (k_hist, k_count, k_write).
#include <cmath>
#include <cstring>
#include <mutex>
#include <unordered_map>

#include <cooperative_groups.h>
#include <cuda.h>

#include "chain_plan.h"
#include "gs_common.cuh"

namespace gs {

namespace cg = cooperative_groups;

namespace {

constexpr int kBins = 2048;
constexpr int kL1Shift = 21;  // level 1: key bits 31..21 (11 bits)
constexpr int kL2Shift = 10;  // level 2: key bits 20..10 (11 bits)
constexpr int kL3Bits = 10;   // level 3: key bits 9..0
constexpr int kScanThreads = 1024;
constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr uint32_t kFull = 0xFFFFFFFFu;

struct SelectState {
  uint32_t prefix;   // key bits fixed so far
  uint32_t k_rem;    // keys still to take inside the prefix
  uint32_t tau;      // the k-th largest key
  uint32_t need_eq;  // keys equal to tau to take
  uint32_t found;    // bit l set when level l found its bin
  uint32_t ncand;    // candidates appended by k_cand
  uint32_t done[3];  // CTAs finished per level (for the last-CTA pick)
  uint32_t prune_key;  // the key below which k_query skips rows (0: none); written once per
                       // query, before k_query, by k_qsample or k_heavy_theta
  uint32_t done_r;     // CTAs finished in k_repair
  uint32_t done_s;     // CTAs finished in k_qsample
  uint32_t open;       // k_query_bits left the whole query to the kernel behind it
};

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

__device__ __forceinline__ uint32_t key_of(float v) { return __float_as_uint(v) & 0x7FFFFFFFu; }

// The hash arithmetic of k_query and k_qsample, without compares.
// For s < 2^62 - 1, s mod p is s - p when s >= p and s otherwise; s >= p exactly when bit 61
// of s + 1 is set, and then s - p = (s + 1) - 2^61 = (s + 1) & p.  So for s < 2p:
//   s mod p = (s + ((s + 1) >> 61)) & p.
__device__ __forceinline__ uint64_t reduce61(uint64_t s) { return (s + ((s + 1) >> 61)) & kP61; }

// x + a mod p for x, a < p (the incremental form of the hash): the same value as step61.
__device__ __forceinline__ uint64_t step61_nb(uint64_t x, uint64_t a) { return reduce61(x + a); }

// (a*i + b) mod p for a, b < p and i < 2^32: the same value as affine61.  The sum of the
// partial products is below 3 * 2^61; one fold leaves it at most p + 2, then reduce61.
__device__ __forceinline__ uint64_t affine61_nb(uint64_t a, uint64_t b, uint32_t i) {
  const uint64_t p0 = (uint64_t)(uint32_t)a * i;
  const uint64_t p1 = (uint64_t)(uint32_t)(a >> 32) * i;
  const uint64_t s = (p1 >> 29) + ((p1 & ((1ull << 29) - 1)) << 32) + fold61(p0) + b;
  return reduce61(fold61(s));
}

// Warp-aggregated shared-memory histogram update; every lane of the warp must call it.
__device__ __forceinline__ void hist_add(uint32_t* sh, uint32_t bin) {
  const uint32_t peers = __match_any_sync(kFull, bin);
  const int leader = __ffs(peers) - 1;
  if (bin != kNone && (int)(threadIdx.x & 31) == leader) atomicAdd(&sh[bin], (uint32_t)__popc(peers));
}

__device__ __forceinline__ void hist_flush(const uint32_t* sh, uint32_t* hist, int nbins) {
  __syncthreads();
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) {
    const uint32_t n = sh[b];
    if (n) atomicAdd(&hist[b], n);
  }
}

// Exclusive scan of one uint32 per thread across the block; *total gets the block sum.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t warp_sums[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = (blockDim.x + 31) >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < nwarps ? warp_sums[lane] : 0u;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, w, o);
      if (lane >= o) w += y;
    }
    warp_sums[lane] = w;
  }
  __syncthreads();
  const uint32_t off = warp ? warp_sums[warp - 1] : 0u;
  *total = warp_sums[nwarps - 1];
  __syncthreads();
  return off + x - v;
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// The whole block finds the bin holding the k_rem-th largest key, scanning from the top bin.
// Histogram values are read past L1 (they were completed by other CTAs' atomics).
__device__ void pick_bins(const uint32_t* hist, int nbits, SelectState* st, int level, uint32_t k_init) {
  const int nbins = 1 << nbits;
  const uint32_t k_rem = level == 0 ? k_init : __ldcg(&st->k_rem);
  const uint32_t prefix = level == 0 ? 0u : __ldcg(&st->prefix);
  const uint32_t found = level == 0 ? 0u : __ldcg(&st->found);
  const int per = (nbins + blockDim.x - 1) / blockDim.x;
  const int r0 = threadIdx.x * per;  // positions counted from the top bin
  uint32_t local = 0;
  for (int t = 0; t < per; ++t) {
    const int rp = r0 + t;
    if (rp < nbins) local += __ldcg(&hist[nbins - 1 - rp]);
  }
  uint32_t total;
  uint32_t cum = block_excl_scan(local, &total);
  for (int t = 0; t < per; ++t) {
    const int rp = r0 + t;
    if (rp >= nbins) break;
    const int bin = nbins - 1 - rp;
    const uint32_t cnt = __ldcg(&hist[bin]);
    if (cum < k_rem && cum + cnt >= k_rem) {
      const uint32_t p = (prefix << nbits) | (uint32_t)bin;
      st->prefix = p;
      st->k_rem = k_rem - cum;
      st->found = found | (1u << level);
      if (level == 2) {
        st->tau = p;
        st->need_eq = k_rem - cum;
      }
    }
    cum += cnt;
  }
}

// Called by every CTA after its histogram atomics: the last CTA to arrive does the pick.
__device__ __forceinline__ void last_block_pick(const uint32_t* hist, int nbits, SelectState* st, int level,
                                                uint32_t k_init, uint32_t* counter = nullptr) {
  __shared__ uint32_t am_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0)
    am_last = (atomicAdd(counter ? counter : &st->done[level], 1u) == gridDim.x - 1) ? 1u : 0u;
  __syncthreads();
  if (am_last) {
    __threadfence();
    pick_bins(hist, nbits, st, level, k_init);
  }
}

template <int R>
__device__ __forceinline__ float median_of(float (&v)[R]) {
#pragma unroll
  for (int i = 0; i < R; ++i) {
#pragma unroll
    for (int j = 0; j + 1 < R - i; ++j) {
      const float lo = fminf(v[j], v[j + 1]), hi = fmaxf(v[j], v[j + 1]);
      v[j] = lo;
      v[j + 1] = hi;
    }
  }
  if (R & 1) return v[R / 2];
  return 0.5f * (v[R / 2 - 1] + v[R / 2]);
}

// The i-th output (i = 0, 1, ...) of the splitmix64 stream seeded with `seed`: the state after
// i + 1 increments of the golden-ratio constant, mixed (Steele, Lea and Flood, 2014).
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t i) {
  uint64_t z = seed + (i + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Composite key of HEAVYMIX.  Members of H = {i : est_i^2 >= theta} get 0x80000000 | bits(|est_i|):
// all of H ranks above all of NH, and inside H by |est|.  Members of NH get 0x7FFFFFFF - xi_i,
// xi_i = the top 31 bits of splitmix64_at(fill_seed, i): the largest NH keys are the NH
// coordinates with the smallest xi, a uniformly random subset (rand_l(NH)).  The top-k of these
// keys (ties to the smaller index) is H plus k - |H| random coordinates of NH when |H| < k, and
// the k largest |est| of H otherwise.
__device__ __forceinline__ uint32_t heavy_key(float e, double theta, uint64_t fill_seed, uint64_t i) {
  const double e2 = (double)e * (double)e;  // exact
  return e2 >= theta ? (0x80000000u | key_of(e)) : 0x7FFFFFFFu - (uint32_t)(splitmix64_at(fill_seed, i) >> 33);
}

struct QueryParams {
  const float* T;     // merged table [r][c]
  float* est;         // [d]
  uint32_t* hist;     // level-1 histogram
  SelectState* st;
  int64_t d;
  uint32_t k;
  int32_t r;
  uint32_t c, cmask;
  uint64_t cinv;      // bucket_inverse(c)
  int32_t vec;        // est 16-byte aligned
  int32_t pick;       // the last CTA picks the level-1 bin from the histogram of the keys
  int32_t prune;      // skip rows below st->prune_key (estimate internal to the workspace)
  int32_t if_open;    // k_query_quads (HEAVYMIX: k_query) is launched behind k_query_bits and runs only where
                      // that kernel left the query to it (st->open)
  uint32_t* keys;     // HEAVYMIX: also store each coordinate's composite key here, and build the
                      // level-1 histogram (and pick) on those keys instead of |est|
  const double* theta;  // HEAVYMIX: the threshold l2sq / k of H
  uint64_t fill_seed;   // HEAVYMIX: the seed of the random fill
  HashCoeffs h;
  HashCoeffs h8;        // 8 a, 8 b, 8 a', 8 b' of every row
  uint64_t qa[GS_MAX_ROWS / 2 + 1][3];  // 8 (t a mod p), t = 1, 2, 3, of the first rows
};

// The low word for coordinate t of a quad, from its first coordinate.
__device__ __forceinline__ uint32_t quad_lo(Rot y, const uint64_t (&step)[3], int t) {
  return t == 0 ? y.lo : rot_add_lo(y, step[t - 1]);
}

// The signed cell of row j for coordinate i.
__device__ __forceinline__ float signed_cell(const QueryParams& prm, int j, uint32_t i) {
  const uint32_t x = rot_at_lo(prm.h8.a[j], prm.h8.b[j], i), y = rot_at_lo(prm.h8.a2[j], prm.h8.b2[j], i);
  return apply_sign(__ldg(prm.T + (size_t)j * prm.c + rot_bucket(x, prm.cmask)), rot_signbit(y));
}

// Row pruning.  With f = r/2 + 1: if at least f of a coordinate's r signed cells are < t and
// at least f are > -t, then -t < est < t.  For odd r the median is the f-th smallest and the
// f-th largest value; for even r the two middle values are the f-th smallest and the f-th
// largest, and the fp32 mean of two values in (-t, t) stays inside (rounding is monotone and
// twice an fp32 value is exact).  So a coordinate can stop reading rows as soon as both counts
// reach f: its |est| < t, and it cannot be among the top k when t is at most the k-th largest
// |est|.  Rows are read in order; the first f always, each later one only while the coordinate
// is undecided.  A cell with |v| < t counts on both sides, so f of those settle it after the
// first f rows; one cell outside (-t, t) among them costs one more row, not all of them.
// The prune key t is computed by this query itself before k_query runs (k_qsample: from the
// full estimate of a strided sample of coordinates; HEAVYMIX: from its threshold) and kept in
// the query's own selection state, so every CTA of k_query and k_repair reads the same value.
// It is a level-1 bin edge: whether it was safe is then exactly whether the level-1 pick
// lands in its bin or above, which k_repair checks.
// A coordinate that stopped early stores the marker -((32 g + n) * 2^-149): n = the rows whose
// cells it examined (f <= n < r), g = how many of those cells it read from the table (g = n
// when every examined cell is read).  It is a key in level-1 bin 0 that k_repair recognises
// and the measurement can count.
constexpr uint32_t kPrunedBits = 0x80000000u;  // sign bit; the low bits hold n and g

__device__ __forceinline__ uint32_t pruned_marker(int examined, int gathered) {
  return kPrunedBits | ((uint32_t)gathered << 5) | (uint32_t)examined;
}

__device__ __forceinline__ bool is_pruned(uint32_t bits) { return bits - (kPrunedBits + 1u) < 0x3FFu; }

// Counts of a coordinate's cells below t (lt) and above -t (gt), on keys: |v| < t is
// key_of(v) < pk; a NaN counts on neither side.
__device__ __forceinline__ void tally(float v, uint32_t pk, int& lt, int& gt) {
  const uint32_t b = __float_as_uint(v), key = b & 0x7FFFFFFFu;
  const bool inside = key < pk;
  const bool number = key <= 0x7F800000u;
  lt += (inside || (number && (b >> 31))) ? 1 : 0;
  gt += (inside || (number && !(b >> 31))) ? 1 : 0;
}

__device__ __forceinline__ uint32_t prune_key_of(const QueryParams& prm) {
  return prm.prune ? __ldcg(&prm.st->prune_key) : 0u;
}

__device__ __forceinline__ void store_est(const QueryParams& prm, int64_t i0, int tmax,
                                          const float (&m)[4]) {
  if (prm.vec && tmax == 4) {
    *reinterpret_cast<float4*>(prm.est + i0) = make_float4(m[0], m[1], m[2], m[3]);
  } else {
    for (int t = 0; t < tmax; ++t) prm.est[i0 + t] = m[t];
  }
}

// ---- the query ----------------------------------------------------------------------------

// Fast path: R rows known at compile time, c a power of two.  A thread takes four consecutive
// coordinates; their hash values after the first come from the incremental form.
// HM: HEAVYMIX mode (prm.keys set): each coordinate's composite key is stored and histogrammed.
// Up to 7 rows the register budget keeps four CTAs per SM (no spills at 64 registers).
template <int R, bool HM = false>
__global__ void __launch_bounds__(kBlock, R <= 7 ? 4 : 1) k_query(const __grid_constant__ QueryParams prm) {
  grid_begin();
  if (HM && prm.if_open && __ldcg(&prm.st->open) == 0u) return;
  __shared__ uint32_t sh[kBins];
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const int64_t d = prm.d, nq = (d + 3) / 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  const uint32_t pk = prune_key_of(prm);
  const double theta = HM ? __ldcg(prm.theta) : 0.0;
  constexpr int kF = R / 2 + 1;  // rows that bound the median
  for (int64_t q0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); q0 < nq; q0 += stride) {
    const int64_t q = q0 + lane;
    const int64_t i0 = q * 4;
    const int tmax = q < nq ? (d - i0 < 4 ? (int)(d - i0) : 4) : 0;
    float m[4] = {0.f, 0.f, 0.f, 0.f};
    uint32_t hk[4] = {0u, 0u, 0u, 0u};
    if (tmax > 0) {
      float v[4][R];
#pragma unroll
      for (int j = 0; j < kF; ++j) {
        uint64_t x = affine61_nb(prm.h.a[j], prm.h.b[j], (uint32_t)i0);
        uint64_t y = affine61_nb(prm.h.a2[j], prm.h.b2[j], (uint32_t)i0);
        const float* row = prm.T + (size_t)j * prm.c;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          v[t][j] = 0.f;
          if (t < tmax) {
            v[t][j] = apply_sign(__ldg(row + ((uint32_t)x & prm.cmask)), signbit_of(y));
            x = step61_nb(x, prm.h.a[j]);
            y = step61_nb(y, prm.h.a2[j]);
          }
        }
      }
      // the later rows, each only while the coordinate is undecided
      int lt[4], gt[4], rows[4];
      bool done[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        lt[t] = 0;
        gt[t] = 0;
#pragma unroll
        for (int j = 0; j < kF; ++j) tally(v[t][j], pk, lt[t], gt[t]);
        rows[t] = kF;
        done[t] = pk != 0u && lt[t] >= kF && gt[t] >= kF;
      }
#pragma unroll
      for (int j = kF; j < R; ++j) {
        uint64_t x = affine61_nb(prm.h.a[j], prm.h.b[j], (uint32_t)i0);
        uint64_t y = affine61_nb(prm.h.a2[j], prm.h.b2[j], (uint32_t)i0);
        const float* row = prm.T + (size_t)j * prm.c;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          v[t][j] = 0.f;
          if (t < tmax) {
            if (!done[t]) {
              v[t][j] = apply_sign(__ldg(row + ((uint32_t)x & prm.cmask)), signbit_of(y));
              tally(v[t][j], pk, lt[t], gt[t]);
              ++rows[t];
            }
            x = step61_nb(x, prm.h.a[j]);
            y = step61_nb(y, prm.h.a2[j]);
          }
        }
        if (j + 1 < R) {
#pragma unroll
          for (int t = 0; t < 4; ++t) done[t] = done[t] || (pk != 0u && lt[t] >= kF && gt[t] >= kF);
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t)
        m[t] = done[t] ? __uint_as_float(pruned_marker(rows[t], rows[t])) : median_of<R>(v[t]);
      store_est(prm, i0, tmax, m);
      if (HM) {
#pragma unroll
        for (int t = 0; t < 4; ++t)
          hk[t] = heavy_key(done[t] ? 0.f : m[t], theta, prm.fill_seed, (uint64_t)(i0 + t));
        if (tmax == 4) {
          *reinterpret_cast<uint4*>(prm.keys + i0) = make_uint4(hk[0], hk[1], hk[2], hk[3]);
        } else {
          for (int t = 0; t < tmax; ++t) prm.keys[i0 + t] = hk[t];
        }
      }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t)
      hist_add(sh, t < tmax ? ((HM ? hk[t] : key_of(m[t])) >> kL1Shift) : kNone);
  }
  hist_flush(sh, prm.hist, kBins);
  if (prm.pick) last_block_pick(prm.hist, 11, prm.st, 0, prm.k);
}

// ---- the query along a walk that serves two rows ---------------------------------------------
// Where the table is too large for k_query_bits, or every estimate is wanted, the query is bound by
// its reads of table cells, one sector request from L1 to L2 each.  A walk along which two rows keep
// their buckets (PairShape in chain_plan.h) needs a new cell of these rows for about a quarter of the
// coordinates only: the inner row's cell stays in a register, the outer row's in shared memory, one
// slot per inner step.  Each lane holds one coordinate; the hash values move by constant steps.
// PRUNE: only the first kF rows are read here; the coordinates that they do not settle are queued
// per warp with the cells read, and resolved 32 at a time, so that the later rows' work is done with
// full warps.
// Query in ms, k_query / here: all rows, d = 25,557,032, r = 5, c = 2^18 0.443 / 0.403; pruning, d =
// 138,357,544, r = 7, c = 2^20 2.26 / 1.81, d = 83,311,104, r = 5, c = 2^21 1.01 / 0.83.  The walk's own
// instructions now take about as long as the reads that are left; without the second coordinate in
// flight the first of these took 0.423.
constexpr int kWalkMaxRows = 9;
constexpr int kWalkSlots = 8;  // inner steps at most

struct WalkRow {
  uint64_t a8, b8, a28, b28;   // 8 times the hash coefficients
  uint64_t sa8, sa28;          // one inner step
  uint64_t ja8[2], ja28[2];    // from the last inner step of a round to the next round: after inner_steps
                               // steps, and after one fewer
  const float* cells;
};

struct WalkParams {
  uint32_t inner, outer;
  int32_t inner_steps, outer_steps;
  uint32_t tiles;              // CTAs across the inner stride
  WalkRow row[kWalkMaxRows];   // the inner row, the outer row, the others
};

template <int R, bool PRUNE>
__global__ void __launch_bounds__(kBlock, R <= 7 ? 3 : 2) k_query_walk(const __grid_constant__ QueryParams prm,
                                                                      const __grid_constant__ WalkParams wk) {
  grid_begin();
  constexpr int kF = R / 2 + 1;
  constexpr int NR = PRUNE ? kF : R;
  constexpr int kEntry = kF + 1;
  __shared__ uint32_t sh[kBins];
  __shared__ float slot_cell[kWalkSlots][kBlock];
  __shared__ uint32_t slot_place[kWalkSlots][kBlock];
  __shared__ uint32_t queues[PRUNE ? kBlock / 32 : 1][PRUNE ? kEntry : 1][64];
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const uint32_t below = (1u << lane) - 1u;
  const uint32_t d = (uint32_t)prm.d, S0 = wk.inner, S1 = wk.outer;
  const uint32_t pk = PRUNE ? prune_key_of(prm) : 0u;
  const uint32_t seg = blockIdx.x / wk.tiles;
  const uint32_t base = (blockIdx.x - seg * wk.tiles) * kBlock + threadIdx.x;
  const int64_t start = (int64_t)seg * wk.outer_steps * S1 + base;
  const bool on = base < S0 && start < prm.d;
  uint32_t i = on ? (uint32_t)start : 0u;
  Rot x[NR], y[NR];
#pragma unroll
  for (int s = 0; s < NR; ++s) {
    x[s] = rot_at(wk.row[s].a8, wk.row[s].b8, i);
    y[s] = rot_at(wk.row[s].a28, wk.row[s].b28, i);
  }
  uint32_t (*queue)[64] = queues[PRUNE ? threadIdx.x >> 5 : 0];
  uint32_t queued = 0;  // the same in every lane of the warp
  uint32_t zeros = 0;   // this lane's markers: keys of bin 0
  const auto drain = [&](uint32_t n) {
    uint32_t bin = kNone;
    if ((uint32_t)lane < n) {
      const uint32_t at = queued + lane, c = queue[0][at];
      float v[R];
      int lt = 0, gt = 0, rows = kF;
#pragma unroll
      for (int j = 0; j < kF; ++j) {
        v[j] = __uint_as_float(queue[1 + j][at]);
        tally(v[j], pk, lt, gt);
      }
      bool done = pk != 0u && lt >= kF && gt >= kF;
#pragma unroll
      for (int j = kF; j < R; ++j) {
        v[j] = 0.f;
        if (!done) {
          v[j] = signed_cell(prm, j, c);
          tally(v[j], pk, lt, gt);
          ++rows;
        }
        if (j + 1 < R) done = done || (pk != 0u && lt >= kF && gt >= kF);
      }
      const float m = done ? __uint_as_float(pruned_marker(rows, rows)) : median_of<R>(v);
      prm.est[c] = m;
      if (done) ++zeros;
      else bin = key_of(m) >> kL1Shift;
    }
    hist_add(sh, bin);
  };
  float cell0 = 0.f;
  uint32_t place0 = 0xFFFFFFFFu;
  uint32_t round = i;  // the coordinate at m = 0
  int m = 0, n = 0;
  bool live = on;
  // A coordinate whose cells are on their way.  Two are kept, so that the reads of one overlap the
  // examination of the other; nothing here waits for a cell before the next one's reads are out.
  struct Flight {
    float raw[NR];
    uint32_t i, m, signs;
    bool held, moved, fresh;  // a coordinate at all; the inner row, the outer row in a new bucket
  };
  // reads the cells of the walk's coordinate, then moves the walk to the next one
  const auto fetch = [&](Flight& f) {
    f.held = live;
    if (!live) return;
    f.i = i;
    f.m = (uint32_t)m;
#pragma unroll
    for (int s = 2; s < NR; ++s) f.raw[s] = __ldg(wk.row[s].cells + rot_bucket(x[s].lo, prm.cmask));
    const uint32_t p0 = (x[0].lo >> 3) & prm.cmask, p1 = (x[1].lo >> 3) & prm.cmask;
    f.moved = p0 != place0;
    if (f.moved) {
      place0 = p0;
      f.raw[0] = __ldg(wk.row[0].cells + ((p0 - 1u) & prm.cmask));
    }
    f.fresh = n == 0 || slot_place[m][threadIdx.x] != p1;
    if (f.fresh) {
      f.raw[1] = __ldg(wk.row[1].cells + ((p1 - 1u) & prm.cmask));
      slot_place[m][threadIdx.x] = p1;
    }
    f.signs = 0;
#pragma unroll
    for (int s = 0; s < NR; ++s) f.signs |= (rot_signbit(y[s].lo) >> 31) << s;
    // the next inner step, or the next round; m * S0 + base = i - round + base
    const bool inside = i - round + base + S0 < S1 && i + S0 < d;
    const bool full = m == wk.inner_steps - 1;
    if (inside) {
      i += S0;
      ++m;
    } else {
      // where the vector ends before the round does, the next round lies beyond it as well
      i = round + S1;
      round = i;
      m = 0;
      ++n;
      live = n < wk.outer_steps && i < d;
    }
#pragma unroll
    for (int s = 0; s < NR; ++s) {
      const WalkRow& r = wk.row[s];
      x[s] = rot_add(x[s], inside ? r.sa8 : full ? r.ja8[0] : r.ja8[1]);
      y[s] = rot_add(y[s], inside ? r.sa28 : full ? r.ja28[0] : r.ja28[1]);
    }
  };
  const auto examine = [&](Flight& f) {
    bool open = false;
    uint32_t bin = kNone;
    float v[R];
#pragma unroll
    for (int s = 0; s < NR; ++s) v[s] = 0.f;
    if (f.held) {
      if (f.moved) cell0 = f.raw[0];
      v[0] = cell0;
      if (f.fresh) slot_cell[f.m][threadIdx.x] = f.raw[1];  // a slot serves again one round later
      else f.raw[1] = slot_cell[f.m][threadIdx.x];
#pragma unroll
      for (int s = 1; s < NR; ++s) v[s] = f.raw[s];
#pragma unroll
      for (int s = 0; s < NR; ++s) v[s] = apply_sign(v[s], (f.signs >> s) << 31);
      if (PRUNE) {
        int lt = 0, gt = 0;
#pragma unroll
        for (int s = 0; s < NR; ++s) tally(v[s], pk, lt, gt);
        open = pk == 0u || lt < kF || gt < kF;
        if (!open) {
          prm.est[f.i] = __uint_as_float(pruned_marker(kF, kF));
          ++zeros;
        }
      } else {
        float t[R];
#pragma unroll
        for (int s = 0; s < R; ++s) t[s] = v[s];
        const float e = median_of<R>(t);
        prm.est[f.i] = e;
        bin = key_of(e) >> kL1Shift;
      }
    }
    if (PRUNE) {
      const uint32_t who = __ballot_sync(kFull, open);
      if (open) {
        const uint32_t at = queued + __popc(who & below);
        queue[0][at] = f.i;
#pragma unroll
        for (int j = 0; j < kF; ++j) queue[1 + j][at] = __float_as_uint(v[j]);
      }
      queued += __popc(who);
      __syncwarp();
      if (queued >= 32) {
        queued -= 32;
        drain(32);
        __syncwarp();
      }
    } else {
      hist_add(sh, bin);
    }
  };
  Flight f0, f1;
  fetch(f0);
  while (__any_sync(kFull, f0.held)) {
    fetch(f1);
    examine(f0);
    fetch(f0);
    examine(f1);
  }
  if (PRUNE) {
    const uint32_t n_left = queued;
    queued = 0;
    if (n_left) drain(n_left);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) zeros += __shfl_down_sync(kFull, zeros, o);
    if (lane == 0 && zeros) atomicAdd(&sh[0], zeros);
  }
  hist_flush(sh, prm.hist, kBins);
  if (prm.pick) last_block_pick(prm.hist, 11, prm.st, 0, prm.k);
}

// ---- the pruning query with the first rows classified in shared memory ---------------------
// The settle rule needs, for each of the first f = r/2 + 1 cells of a coordinate, only which side
// of the prune key t its value lies on: whether it counts below t, above -t, or both (|T| < t: the
// cell is inside).  That takes two bits per table cell: one says whether the cell is inside, the
// other, for the others, on which side it lies; the coordinate's sign hash swaps the sides.
// Where the bits of the first f rows fit in shared memory, k_pbits writes them once per query and
// k_query_bits looks them up instead of reading those cells from L2.  A coordinate that settles
// within the first f rows then reads no cell at all; one that examines later rows reads those
// cells as k_query does; one that does not settle reads every cell for its full median.  The rows
// examined, the stops and the estimates are the same as k_query's, for tables without NaN (a NaN cell
// counts on the side of its sign bit here and on neither there).
//
// The kernel sorts its coordinates by the work that they need, so that warps stay full.
//   1. f rows settle a coordinate exactly when all f cells are inside, whatever the signs: four
//      coordinates per lane, only the buckets of the first f rows, whose hash comes from a form
//      that needs few instructions (rot_add).  The others are queued, per warp.
//   2. With one cell of the first f outside, the next row settles a coordinate when its cell is
//      inside, again whatever the signs: 32 such coordinates at a time, one per lane, one bucket and
//      one cell read each.
//   3. What is left is resolved from its signs and all further rows, 32 coordinates at a time.
// Integer instructions bound it.  d = 25,557,032, r = 5, c = 2^18: 0.098 ms, and 0.110 in HEAVYMIX
// mode (which evaluates the fill order of every coordinate); one kernel for all coordinates, four per
// lane, took 0.267, and 0.344 with k_query in HEAVYMIX mode.  Part 3 without part 2 takes 0.145.
//
// The sorting pays while parts 1 and 2 settle enough coordinates; where most are left for part 3 (a large k,
// many rows, few columns: the prune key lies within the cells' noise), evaluating every row of four
// coordinates per lane from the start is the better order (k_query_quads).  Every CTA takes the same sample of
// the inside bits, and the query is left to that kernel, launched behind, where more than kMostlyOpen of the
// coordinates would be left.  Query with its selection in us, sorted / quads,
// d = 25.6M: r = 7, c = 2^16, k = d/1000, d/100, d/30, d/10 (shares left 0.19, 0.52, 0.71, 0.80) 277 / 440,
// 456 / 478, 599 / 533, 652 / 551; r = 16, c = 2^14, k = d/1000 (0.97) 1450 / 1127.  The line is the one with the
// least loss over 610 shapes (r 3 to 16, c 2^10 to 2^18, k d/10000 to d/3).  With many rows and few cells inside,
// nearly every coordinate reads every cell; the quads' registers spill, and one coordinate per lane is the
// faster order again where the cells come from L2 (r = 16, k = d/3, 0.22 of the cells inside: c = 2^14 1781 /
// 1951, c = 2^16 1696 / 1990, but c = 2^10 1566 / 1270).
constexpr uint32_t kBitsBytes = 192u << 10;   // dynamic shared memory for the bits

constexpr int kBitsBlock = 1024;              // one CTA of 32 warps per SM
constexpr float kMostlyOpen = 0.55f;          // share left for part 3 from which quads are faster
// ... and in HEAVYMIX mode k_query, which reads the cells from the start: where its threshold leaves most
// coordinates open, they need every cell.  k_query has more to spill for many rows.
__host__ __device__ constexpr float heavy_open(int r) { return r < 8 ? 0.6f : r < 11 ? 0.75f : r < 16 ? 0.87f : 1.f; }
// Queue entries per warp.  Queue 2 grows from the front, queue 3 from the back; each keeps at most
// 31 entries from one grid stride to the next, which adds at most 128.
constexpr int kQueue = 192;

// 8 (n a mod p) of the first r/2 + 1 rows for the n coordinates of one grid stride.
struct GridSteps {
  uint64_t a[GS_MAX_ROWS / 2 + 1];
};

// The bits of the first kf rows: kf * c / 32 words that tell inside from outside, then as many that
// tell the side of an outside cell (set: T <= -t).  Bit n mod 32 of word n / 32 of a row belongs to
// the cell of bucket n - 1 mod c: its place (x + 1) mod c is what the hash gives first.
__global__ void __launch_bounds__(kBlock) k_pbits(const float* __restrict__ T, uint32_t c, int64_t nwords,
                                                  const SelectState* st, uint32_t* __restrict__ words) {
  grid_begin();
  const uint32_t pk = __ldcg(&st->prune_key);
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x / 32);
  constexpr int kN = 4;  // words of a warp in flight
  for (int64_t w0 = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); w0 < nwords; w0 += kN * warps) {
    float v[kN];
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      const uint32_t w = (uint32_t)(w0 + u * warps);
      const uint32_t j = w / (c / 32), n = (w - j * (c / 32)) * 32 + lane;
      v[u] = w0 + u * warps < nwords ? __ldg(T + (size_t)j * c + ((n - 1u) & (c - 1u))) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kN; ++u) {
      const uint32_t in = __ballot_sync(kFull, key_of(v[u]) < pk);
      const uint32_t side = __ballot_sync(kFull, (__float_as_uint(v[u]) >> 31) != 0u);
      if (w0 + u * warps < nwords && lane < 2) words[w0 + u * warps + (lane ? nwords : 0)] = lane ? side : in;
    }
  }
}

// A coordinate i from its signs: its first kF cells by their bits, the later rows from the table
// while it is undecided, and its full median when it does not settle.  Returns the marker (settled)
// or the estimate: the value alone does not tell them apart, an estimate may have a marker's bits.
template <int R>
__device__ __forceinline__ float resolve(const QueryParams& prm, const uint32_t* sbits, uint32_t i, uint32_t pk,
                                         bool& settled) {
  constexpr int kF = R / 2 + 1;
  const uint32_t per_row = prm.c / 32;
  uint32_t cell[kF];  // bucket of each of the first kF rows, sign bit of the cell in bit 31
  int lt = 0, gt = 0, rows = kF;
#pragma unroll
  for (int j = 0; j < kF; ++j) {
    const uint32_t x = rot_at_lo(prm.h8.a[j], prm.h8.b[j], i), y = rot_at_lo(prm.h8.a2[j], prm.h8.b2[j], i);
    const uint32_t w = j * per_row + ((x >> 8) & (per_row - 1u));  // place (x >> 3) mod c
    const uint32_t in = __funnelshift_r(sbits[w], 0u, x >> 3) & 1u;
    const uint32_t below = (__funnelshift_r(sbits[kF * per_row + w], 0u, x >> 3) ^ ~(y >> 3)) & 1u;
    lt += (int)(in | below);
    gt += (int)(in | (below ^ 1u));
    cell[j] = rot_bucket(x, prm.cmask) | rot_signbit(y);
  }
  bool done = pk != 0u && lt >= kF && gt >= kF;
  float v[R];
#pragma unroll
  for (int j = kF; j < R; ++j) {
    v[j] = 0.f;
    if (!done) {
      v[j] = signed_cell(prm, j, i);
      tally(v[j], pk, lt, gt);
      ++rows;
    }
    if (j + 1 < R) done = done || (pk != 0u && lt >= kF && gt >= kF);
  }
  settled = done;
  if (done) return __uint_as_float(pruned_marker(rows, rows - kF));
#pragma unroll
  for (int j = 0; j < kF; ++j)
    v[j] = apply_sign(__ldg(prm.T + (size_t)j * prm.c + (cell[j] & 0x7FFFFFFFu)), cell[j] & 0x80000000u);
  return median_of<R>(v);
}

// The share of the coordinates that parts 1 and 2 leave open, p of the cells being inside.
template <int R>
__device__ __forceinline__ float left_open(float p) {
  constexpr int kF = R / 2 + 1;
  float few = 1.f;  // p^(kF - 1)
#pragma unroll
  for (int j = 1; j < kF; ++j) few *= p;
  return 1.f - few * p - (kF + 1 < R ? kF * few * (1.f - p) * p : 0.f);
}

// The even bits of the result are the low 16 bits of x.
__device__ __forceinline__ uint32_t spread_bits(uint32_t x) {
  x &= 0xFFFFu;
  x = (x | (x << 8)) & 0x00FF00FFu;
  x = (x | (x << 4)) & 0x0F0F0F0Fu;
  x = (x | (x << 2)) & 0x33333333u;
  return (x | (x << 1)) & 0x55555555u;
}

// The pruning query where few coordinates settle early: every row of four consecutive coordinates per
// lane, the first kF by a class of two bits in shared memory (bit 1: the cell counts below t, bit 0: above
// -t; place n of a row at bits 2n, 2n + 1), the later ones from the table while a coordinate is undecided,
// all cells for the full median of one that does not settle.  A kernel of its own: within k_query_bits its
// registers cost the sorted order 3 % (r = 5, d = 25.6M, c = 2^18: 186 -> 192 us).
template <int R>
__global__ void __launch_bounds__(kBitsBlock, 1) k_query_quads(const __grid_constant__ QueryParams prm,
                                                               const uint32_t* __restrict__ words) {
  grid_begin();
  if (__ldcg(&prm.st->open) == 0u) return;
  extern __shared__ uint4 sbits4[];
  uint32_t* classes = reinterpret_cast<uint32_t*>(sbits4);
  __shared__ uint32_t sh[kBins];
  const uint32_t half = (R / 2 + 1) * (prm.c / 32);  // words of one kind of bit
  for (uint32_t w = threadIdx.x; w < half; w += blockDim.x) {
    const uint32_t in = __ldcg(words + w), side = __ldcg(words + half + w);
    const uint32_t below = in | side, above = in | ~side;
    classes[2 * w] = spread_bits(above) | spread_bits(below) << 1;
    classes[2 * w + 1] = spread_bits(above >> 16) | spread_bits(below >> 16) << 1;
  }
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const uint32_t pk = prune_key_of(prm);
  constexpr int kF = R / 2 + 1;
  const uint32_t per_row = prm.c / 16;
  const int64_t d = prm.d, nq = (d + 3) / 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); q0 < nq; q0 += stride) {
    const int64_t q = q0 + (threadIdx.x & 31);
    const int64_t i0 = q * 4;
    const int tmax = q < nq ? (d - i0 < 4 ? (int)(d - i0) : 4) : 0;
    float m[4] = {0.f, 0.f, 0.f, 0.f};
    if (tmax > 0) {
      float v[4][R];
      uint32_t cell[4][kF];  // bucket of each of the first kF rows, sign bit of the cell in bit 31
      uint32_t count[4] = {0u, 0u, 0u, 0u};  // cells below t in bits 0-7, above -t in bits 8-15
      int lt[4], gt[4], rows[4];
      bool done[4];
#pragma unroll
      for (int j = 0; j < kF; ++j) {
        uint64_t x = affine61_nb(prm.h.a[j], prm.h.b[j], (uint32_t)i0);
        uint64_t y = affine61_nb(prm.h.a2[j], prm.h.b2[j], (uint32_t)i0);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          cell[t][j] = 0u;
          if (t < tmax) {
            const uint32_t b = (uint32_t)x & prm.cmask, n = (b + 1u) & prm.cmask;
            const uint32_t cls = (classes[j * per_row + (n >> 4)] >> ((n & 15u) * 2u)) & 3u;
            // a negative sign swaps the two bits; one product puts each where it is counted
            const uint32_t sg = (uint32_t)y & 1u;
            count[t] += ((cls * (sg ? 0x81u : 0x201u)) >> (1u - sg)) & 0x101u;
            cell[t][j] = b | signbit_of(y);
            x = step61_nb(x, prm.h.a[j]);
            y = step61_nb(y, prm.h.a2[j]);
          }
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        lt[t] = (int)(count[t] & 0xFFu);
        gt[t] = (int)(count[t] >> 8);
        rows[t] = kF;
        done[t] = pk != 0u && lt[t] >= kF && gt[t] >= kF;
      }
#pragma unroll
      for (int j = kF; j < R; ++j) {
        uint64_t x = affine61_nb(prm.h.a[j], prm.h.b[j], (uint32_t)i0);
        uint64_t y = affine61_nb(prm.h.a2[j], prm.h.b2[j], (uint32_t)i0);
        const float* row = prm.T + (size_t)j * prm.c;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          v[t][j] = 0.f;
          if (t < tmax) {
            if (!done[t]) {
              v[t][j] = apply_sign(__ldg(row + ((uint32_t)x & prm.cmask)), signbit_of(y));
              tally(v[t][j], pk, lt[t], gt[t]);
              ++rows[t];
            }
            x = step61_nb(x, prm.h.a[j]);
            y = step61_nb(y, prm.h.a2[j]);
          }
        }
        if (j + 1 < R) {
#pragma unroll
          for (int t = 0; t < 4; ++t) done[t] = done[t] || (pk != 0u && lt[t] >= kF && gt[t] >= kF);
        }
      }
#pragma unroll
      for (int j = 0; j < kF; ++j) {
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          v[t][j] = 0.f;
          if (t < tmax && !done[t])
            v[t][j] = apply_sign(__ldg(prm.T + (size_t)j * prm.c + (cell[t][j] & 0x7FFFFFFFu)), cell[t][j] & 0x80000000u);
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t)
        m[t] = done[t] ? __uint_as_float(pruned_marker(rows[t], rows[t] - kF)) : median_of<R>(v[t]);
      store_est(prm, i0, tmax, m);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) hist_add(sh, t < tmax ? (key_of(m[t]) >> kL1Shift) : kNone);
  }
  hist_flush(sh, prm.hist, kBins);
  last_block_pick(prm.hist, 11, prm.st, 0, prm.k);
}

// HM: HEAVYMIX mode (prm.keys set): each coordinate's composite key is stored and histogrammed.
template <int R, bool HM>
__global__ void __launch_bounds__(kBitsBlock, 1) k_query_bits(const __grid_constant__ QueryParams prm,
                                                              const uint32_t* __restrict__ words,
                                                              const __grid_constant__ GridSteps steps) {
  grid_begin();
  extern __shared__ uint4 sbits4[];
  const uint32_t* sbits = reinterpret_cast<const uint32_t*>(sbits4);
  __shared__ uint32_t sh[kBins];
  __shared__ uint32_t queues[kBitsBlock / 32][kQueue];
  constexpr int kF = R / 2 + 1;
  constexpr bool kNextRow = kF + 1 < R;  // a marker names fewer than R rows
  const uint32_t per_row = prm.c / 32;
  const uint32_t half = kF * per_row;  // words of one kind of bit
  // one inside bit per thread, spread over the rows: a sample that every CTA takes alike
  const uint32_t sampled = __ldcg(words + (uint32_t)((uint64_t)threadIdx.x * half / kBitsBlock));
  {
    const uint4* src = reinterpret_cast<const uint4*>(words);
    for (uint32_t w = threadIdx.x; w < half / 2; w += blockDim.x) sbits4[w] = __ldcg(src + w);
  }
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0;
  const float inside = (float)__syncthreads_count((sampled >> (threadIdx.x & 31)) & 1u) * (1.f / kBitsBlock);
  const uint32_t pk = prune_key_of(prm);
  const double theta = HM ? __ldcg(prm.theta) : 0.0;
  const float open = left_open<R>(inside);
  if (prm.if_open && (HM ? open > heavy_open(R) : open > kMostlyOpen && !(R >= 8 && inside < 0.3f && prm.c >= 1u << 14))) {
    if (blockIdx.x == 0 && threadIdx.x == 0) prm.st->open = 1;
    return;
  }
  const int64_t d = prm.d, nq = (d + 3) / 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  const uint32_t below = (1u << lane) - 1u;
  const float settled = __uint_as_float(pruned_marker(kF, 0));
  uint32_t* queue = queues[threadIdx.x >> 5];
  uint32_t n2 = 0, n3 = 0;  // entries in the queues, the same in every lane of the warp
  uint32_t zeros = 0;       // this lane's markers: keys of bin 0
  const auto push3 = [&](bool who, uint32_t i) {
    const uint32_t m = __ballot_sync(kFull, who);
    n3 += __popc(m);
    if (who) queue[kQueue - n3 + __popc(m & below)] = i;
  };
  // the estimate of coordinate i or its marker, and its key in HEAVYMIX
  const auto record = [&](uint32_t i, float m, bool marker) {
    prm.est[i] = m;
    if (HM) {
      const uint32_t key = heavy_key(marker ? 0.f : m, theta, prm.fill_seed, (uint64_t)i);
      prm.keys[i] = key;
      return key >> kL1Shift;
    }
    zeros += marker ? 1u : 0u;
    return marker ? kNone : key_of(m) >> kL1Shift;
  };
  const auto drain3 = [&](bool active) {
    uint32_t bin = kNone;
    if (active) {
      const uint32_t i = queue[kQueue - n3 + lane];
      bool done;
      const float m = resolve<R>(prm, sbits, i, pk, done);
      bin = record(i, m, done);
    }
    hist_add(sh, bin);
  };
  const auto drain2 = [&](bool active) {
    uint32_t i = 0;
    bool open = false;
    if (active) {
      i = queue[n2 + lane];
      const uint32_t x = rot_at_lo(prm.h8.a[kF], prm.h8.b[kF], i);
      open = key_of(__ldg(prm.T + (size_t)kF * prm.c + rot_bucket(x, prm.cmask))) >= pk;
      if (!open) {
        const uint32_t bin = record(i, __uint_as_float(pruned_marker(kF + 1, 1)), true);
        if (HM) atomicAdd(&sh[bin], 1u);
      }
    }
    __syncwarp();  // the entries are read before the queue grows again
    push3(open, i);
  };
  int64_t q0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31);
  Rot x[kF];  // the first coordinate of the lane's quad
#pragma unroll
  for (int j = 0; j < kF; ++j) x[j] = rot_at(prm.h8.a[j], prm.h8.b[j], (uint32_t)((q0 + lane) * 4));
  for (; q0 < nq; q0 += stride) {
    const int64_t q = q0 + lane;
    const int64_t i0 = q * 4;
    const int tmax = q < nq ? (d - i0 < 4 ? (int)(d - i0) : 4) : 0;
    // bit 0: none, at most one of the rows so far has its cell outside
    uint32_t none[4] = {1u, 1u, 1u, 1u}, one[4] = {1u, 1u, 1u, 1u};
#pragma unroll
    for (int j = 0; j < kF; ++j) {
      const uint32_t* row = sbits + j * per_row;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        // the bit of place (n8 >> 3) mod c; the shift takes its amount modulo 32
        const uint32_t n8 = quad_lo(x[j], prm.qa[j], t);
        const uint32_t in = __funnelshift_r(row[(n8 >> 8) & (per_row - 1u)], 0u, n8 >> 3);
        if (kNextRow) one[t] = (one[t] & in) | none[t];
        none[t] &= in;
      }
      x[j] = rot_add(x[j], steps.a[j]);
    }
    uint32_t hk[4];
    if (tmax > 0) {
      const float m[4] = {settled, settled, settled, settled};
      store_est(prm, i0, tmax, m);
      if (HM) {  // the keys of the settled; those of the queued are replaced below
#pragma unroll
        for (int t = 0; t < 4; ++t) hk[t] = heavy_key(0.f, theta, prm.fill_seed, (uint64_t)(i0 + t));
        if (tmax == 4) {
          *reinterpret_cast<uint4*>(prm.keys + i0) = make_uint4(hk[0], hk[1], hk[2], hk[3]);
        } else {
          for (int t = 0; t < tmax; ++t) prm.keys[i0 + t] = hk[t];
        }
      }
    }
    zeros += (uint32_t)tmax;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const bool open = t < tmax && !(none[t] & 1u);
      const bool second = kNextRow && open && (one[t] & 1u);
      if (HM) {
        if (t < tmax && !open) atomicAdd(&sh[hk[t] >> kL1Shift], 1u);  // spread over 1024 bins
      } else if (open) {
        --zeros;
      }
      if (kNextRow) {
        const uint32_t who = __ballot_sync(kFull, second);
        if (second) queue[n2 + __popc(who & below)] = (uint32_t)i0 + t;
        n2 += __popc(who);
      }
      push3(open && !second, (uint32_t)i0 + t);
    }
    __syncwarp();  // the queues, and the markers that the estimates below replace
    while (true) {
      while (n3 >= 32) {
        drain3(true);
        n3 -= 32;
      }
      if (!kNextRow || n2 < 32) break;
      n2 -= 32;
      drain2(true);
      __syncwarp();
    }
    __syncwarp();
  }
  if (kNextRow) {
    const uint32_t n = n2;
    n2 = 0;
    drain2((uint32_t)lane < n);
    __syncwarp();
  }
  while (n3 > 0) {
    const uint32_t n = n3 < 32 ? n3 : 32;
    drain3((uint32_t)lane < n);
    n3 -= n;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) zeros += __shfl_down_sync(kFull, zeros, o);
  if (!HM && lane == 0 && zeros) atomicAdd(&sh[0], zeros);
  hist_flush(sh, prm.hist, kBins);
  last_block_pick(prm.hist, 11, prm.st, 0, prm.k);
}

// Runs after k_query.  If the level-1 pick landed in the prune key's bin or above, the k-th
// largest |est| is at least the prune key and pruning changed nothing the selection sees: the
// kernel returns at once.  Otherwise every stored marker (each pruned coordinate, and any
// genuine estimate with the same bits, which recomputes to itself) gets its full median, the
// level-1 histogram is rebuilt from all estimates into hist_r, and the level-1 pick is made
// again.
template <int R>
__global__ void __launch_bounds__(kBlock) k_repair(const __grid_constant__ QueryParams prm, uint32_t* hist_r) {
  grid_begin();
  const uint32_t pk = __ldcg(&prm.st->prune_key);
  if (pk == 0u || __ldcg(&prm.st->prefix) >= (pk >> kL1Shift)) return;  // uniform over the grid
  __shared__ uint32_t sh[kBins];
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const int64_t d = prm.d;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < d; base += stride) {
    const int64_t i = base + lane;
    uint32_t bin = kNone;
    if (i < d) {
      float e = prm.est[i];
      if (is_pruned(__float_as_uint(e))) {
        float v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = signed_cell(prm, j, (uint32_t)i);
        e = median_of<R>(v);
        prm.est[i] = e;
      }
      bin = key_of(e) >> kL1Shift;
    }
    hist_add(sh, bin);
  }
  hist_flush(sh, hist_r, kBins);
  last_block_pick(hist_r, 11, prm.st, 0, prm.k, &prm.st->done_r);
}

// The prune key of this query, from a fixed strided sample: the first four coordinates of
// every kSampleQuads * 4 (all rows, full median).  The last CTA finds the level-1 bin holding
// the j_target-th largest sampled key and stores its lower edge as st->prune_key (0, i.e. no
// pruning, when that is bin 0 or the sample holds fewer keys).  j_target is set on the host
// well above the sample's expected share of the top k, so that the key lies below the k-th
// largest |est| of the whole estimate except with negligible probability; k_repair makes the
// result exact in that case as well.
constexpr int64_t kSampleQuads = 64;

template <int R>
__global__ void __launch_bounds__(kBlock) k_qsample(const __grid_constant__ QueryParams prm, uint32_t* hist_s,
                                                    uint32_t j_target) {
  grid_begin();
  __shared__ uint32_t sh[kBins];
  __shared__ uint32_t am_last;
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const int64_t d = prm.d, nq = (d + 3) / 4, ns = (nq + kSampleQuads - 1) / kSampleQuads;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  for (int64_t s0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); s0 < ns; s0 += stride) {
    const int64_t sq = s0 + lane;
    const int64_t i0 = sq * kSampleQuads * 4;
    const int tmax = sq < ns ? (d - i0 < 4 ? (int)(d - i0) : 4) : 0;
    float m[4] = {0.f, 0.f, 0.f, 0.f};
    if (tmax > 0) {
      float v[4][R];
#pragma unroll
      for (int j = 0; j < R; ++j) {
        uint64_t x = affine61_nb(prm.h.a[j], prm.h.b[j], (uint32_t)i0);
        uint64_t y = affine61_nb(prm.h.a2[j], prm.h.b2[j], (uint32_t)i0);
        const float* row = prm.T + (size_t)j * prm.c;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          v[t][j] = 0.f;
          if (t < tmax) {
            v[t][j] = apply_sign(__ldg(row + ((uint32_t)x & prm.cmask)), signbit_of(y));
            x = step61_nb(x, prm.h.a[j]);
            y = step61_nb(y, prm.h.a2[j]);
          }
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) m[t] = median_of<R>(v[t]);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) hist_add(sh, t < tmax ? (key_of(m[t]) >> kL1Shift) : kNone);
  }
  hist_flush(sh, hist_s, kBins);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) am_last = (atomicAdd(&prm.st->done_s, 1u) == gridDim.x - 1) ? 1u : 0u;
  __syncthreads();
  if (!am_last) return;
  __threadfence();
  const int per = (kBins + blockDim.x - 1) / blockDim.x;
  const int r0 = threadIdx.x * per;  // positions counted from the top bin
  uint32_t local = 0;
  for (int t = 0; t < per; ++t) {
    if (r0 + t < kBins) local += __ldcg(&hist_s[kBins - 1 - (r0 + t)]);
  }
  uint32_t total;
  uint32_t cum = block_excl_scan(local, &total);
  for (int t = 0; t < per; ++t) {
    const int rp = r0 + t;
    if (rp >= kBins) break;
    const int bin = kBins - 1 - rp;
    const uint32_t cnt = __ldcg(&hist_s[bin]);
    if (cum < j_target && cum + cnt >= j_target) prm.st->prune_key = bin > 0 ? (uint32_t)bin << kL1Shift : 0u;
    cum += cnt;
  }
}

// Request-ceiling probe of the query (measurement aid): the loads of k_query with every row
// read (the same grid, hash buckets and incremental form), without the median, the estimate
// store or the histogram.  Each CTA writes the sum of what it read to out[blockIdx.x], so that
// the loads cannot be dropped.
template <int R>
__global__ void __launch_bounds__(kBlock) k_gather_probe(const __grid_constant__ QueryParams prm, float* out) {
  grid_begin();
  __shared__ float warp_sum[kBlock / 32];
  const int64_t d = prm.d, nq = (d + 3) / 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  float acc = 0.f;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += stride) {
    const int64_t i0 = q * 4;
    const int tmax = d - i0 < 4 ? (int)(d - i0) : 4;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      uint64_t x = affine61(prm.h.a[j], prm.h.b[j], (uint32_t)i0);
      const float* row = prm.T + (size_t)j * prm.c;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (t < tmax) {
          acc += __ldg(row + ((uint32_t)x & prm.cmask));
          x = step61(x, prm.h.a[j]);
        }
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o);
  if ((threadIdx.x & 31) == 0) warp_sum[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < kBlock / 32; ++w) t += warp_sum[w];
    out[blockIdx.x] = t;
  }
}

// c not a power of two: every row of four consecutive coordinates per thread, as k_query without
// pruning.  d = 3,000,017, r = 4, c = 30,011: 53 us (95 with 64-bit remainders and the
// cells of a coordinate sorted in local memory).
template <int R>
__global__ void __launch_bounds__(kBlock, R <= 7 ? 4 : 1) k_query_mod(const __grid_constant__ QueryParams prm) {
  grid_begin();
  __shared__ uint32_t sh[kBins];
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const int64_t d = prm.d, nq = (d + 3) / 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  const bool heavy = prm.keys != nullptr;
  const double theta = heavy ? __ldcg(prm.theta) : 0.0;
  for (int64_t q0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); q0 < nq; q0 += stride) {
    const int64_t q = q0 + lane;
    const int64_t i0 = q * 4;
    const int tmax = q < nq ? (d - i0 < 4 ? (int)(d - i0) : 4) : 0;
    uint32_t key[4] = {0u, 0u, 0u, 0u};
    if (tmax > 0) {
      float v[4][R], m[4];
#pragma unroll
      for (int j = 0; j < R; ++j) {
        uint64_t x = affine61_nb(prm.h.a[j], prm.h.b[j], (uint32_t)i0);
        uint64_t y = affine61_nb(prm.h.a2[j], prm.h.b2[j], (uint32_t)i0);
        const float* row = prm.T + (size_t)j * prm.c;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          v[t][j] = 0.f;
          if (t < tmax) {
            v[t][j] = apply_sign(__ldg(row + bucket_of<false>(x, prm.c, prm.cmask, prm.cinv)), signbit_of(y));
            x = step61_nb(x, prm.h.a[j]);
            y = step61_nb(y, prm.h.a2[j]);
          }
        }
      }
#pragma unroll
      for (int t = 0; t < 4; ++t) m[t] = median_of<R>(v[t]);
      store_est(prm, i0, tmax, m);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        key[t] = heavy ? heavy_key(m[t], theta, prm.fill_seed, (uint64_t)(i0 + t)) : key_of(m[t]);
        if (heavy && t < tmax) prm.keys[i0 + t] = key[t];
      }
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) hist_add(sh, t < tmax ? (key[t] >> kL1Shift) : kNone);
  }
  hist_flush(sh, prm.hist, kBins);
  if (prm.pick) last_block_pick(prm.hist, 11, prm.st, 0, prm.k);
}

// Four float4 of est per thread in flight (kU strides of the grid-stride loop).
constexpr int kU = 4;

__device__ __forceinline__ void load_quads(const float* __restrict__ est, int64_t d, int vec, int64_t q0,
                                           int64_t stride, float (&v)[kU][4], int (&tm)[kU]) {
  const int64_t nq = (d + 3) / 4;
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const int64_t q = q0 + u * stride + lane;
    const int64_t i0 = q * 4;
    tm[u] = q < nq ? (d - i0 < 4 ? (int)(d - i0) : 4) : 0;
    if (vec && tm[u] == 4) {
      const float4 f = __ldcs(reinterpret_cast<const float4*>(est + i0));
      v[u][0] = f.x; v[u][1] = f.y; v[u][2] = f.z; v[u][3] = f.w;
    } else {
#pragma unroll
      for (int t = 0; t < 4; ++t) v[u][t] = t < tm[u] ? est[i0 + t] : 0.f;
    }
  }
}

// ---- selection with candidate lists --------------------------------------------------------

// One pass over est after the level-1 pick.  Keys above the level-1 bin are selected for
// certain: their bit goes into gt_bm.  Keys inside the bin are candidates (index, key): they
// feed the level-2 histogram and are appended to `cand`; the level-2 pick follows.  Both are
// rare (fewer than k keys lie above the bin, and the bin is a narrow band of keys), so the
// common path per key is a mask, a shift and a compare.  Candidates collect in a block-local
// buffer (slots taken with a warp-aggregated shared atomic) that is copied out with one
// global reservation per block; a block whose buffer fills up appends the rest directly
// (warp-aggregated global atomics), which only happens for inputs with many equal keys.
// `src` holds the keys as 32-bit words: the bits of est (kmask drops the sign) or a key array.
constexpr int kCandBuf = 2048;

__device__ __forceinline__ void cand_append(uint32_t i, uint32_t key, uint32_t* sh_n, uint2* sh_cand,
                                            SelectState* st, uint2* __restrict__ cand) {
  const int lane = threadIdx.x & 31;
  uint32_t am = __activemask();
  int leader = __ffs(am) - 1;
  uint32_t base = 0;
  if (lane == leader) base = atomicAdd(sh_n, (uint32_t)__popc(am));
  base = __shfl_sync(am, base, leader);
  const uint32_t slot = base + __popc(am & ((1u << lane) - 1u));
  if (slot < (uint32_t)kCandBuf) {
    sh_cand[slot] = make_uint2(i, key);
    return;
  }
  am = __activemask();
  leader = __ffs(am) - 1;
  uint32_t gbase = 0;
  if (lane == leader) gbase = atomicAdd(&st->ncand, (uint32_t)__popc(am));
  gbase = __shfl_sync(am, gbase, leader);
  cand[gbase + __popc(am & ((1u << lane) - 1u))] = make_uint2(i, key);
}

__global__ void __launch_bounds__(kBlock) k_cand(const float* __restrict__ src, int64_t d, int vec, uint32_t kmask,
                                                 SelectState* st, uint32_t* hist2, uint2* __restrict__ cand,
                                                 uint32_t* gt_bm) {
  grid_begin();
  __shared__ uint32_t sh[kBins];
  __shared__ uint2 sh_cand[kCandBuf];
  __shared__ uint32_t sh_n, sh_base;
  for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0;
  if (threadIdx.x == 0) sh_n = 0;
  __syncthreads();
  const uint32_t b1 = __ldcg(&st->prefix);
  const int64_t nq = (d + 3) / 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  for (int64_t q0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); q0 < nq; q0 += kU * stride) {
    float v[kU][4];
    int tm[kU];
    load_quads(src, d, vec, q0, stride, v, tm);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const uint32_t i0 = (uint32_t)((q0 + u * stride + lane) * 4);
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const uint32_t key = __float_as_uint(v[u][t]) & kmask;
        if (t < tm[u] && (key >> kL1Shift) >= b1) {
          const uint32_t i = i0 + t;
          if ((key >> kL1Shift) > b1) {
            atomicOr(&gt_bm[i >> 5], 1u << (i & 31));
          } else {
            atomicAdd(&sh[(key >> kL2Shift) & (kBins - 1)], 1u);
            cand_append(i, key, &sh_n, sh_cand, st, cand);
          }
        }
      }
    }
  }
  __syncthreads();
  const uint32_t n = sh_n < (uint32_t)kCandBuf ? sh_n : (uint32_t)kCandBuf;
  if (threadIdx.x == 0) sh_base = n ? atomicAdd(&st->ncand, n) : 0u;
  __syncthreads();
  for (uint32_t t = threadIdx.x; t < n; t += blockDim.x) cand[sh_base + t] = sh_cand[t];
  hist_flush(sh, hist2, kBins);
  last_block_pick(hist2, 11, st, 1, 0);
}

// Level-3 histogram of the candidates that match the 22-bit prefix; the last pick gives tau.
__global__ void __launch_bounds__(kBlock) k_cand_hist3(const uint2* __restrict__ cand, SelectState* st,
                                                       uint32_t* hist3) {
  grid_begin();
  constexpr int kN3 = 1 << kL3Bits;
  __shared__ uint32_t sh[kN3];
  for (int b = threadIdx.x; b < kN3; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const uint32_t n = __ldcg(&st->ncand);
  const uint32_t p22 = __ldcg(&st->prefix);
  const uint32_t stride = gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  for (uint32_t t0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); t0 < n; t0 += stride) {
    const uint32_t t = t0 + lane;
    uint32_t bin = kNone;
    if (t < n) {
      const uint32_t key = cand[t].y;
      if ((key >> kL2Shift) == p22) bin = key & (uint32_t)(kN3 - 1);
    }
    if (__any_sync(kFull, bin != kNone)) hist_add(sh, bin);
  }
  hist_flush(sh, hist3, kN3);
  last_block_pick(hist3, kL3Bits, st, 2, 0);
}

// Candidates above tau into gt_bm, candidates equal to tau into eq_bm.
__global__ void __launch_bounds__(kBlock) k_cand_mark(const uint2* __restrict__ cand, const SelectState* st,
                                                      uint32_t* gt_bm, uint32_t* eq_bm) {
  grid_begin();
  const uint32_t n = __ldcg(&st->ncand);
  const uint32_t tau = __ldcg(&st->tau);
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const uint2 c = cand[t];
    if (c.y > tau) atomicOr(&gt_bm[c.x >> 5], 1u << (c.x & 31));
    else if (c.y == tau) atomicOr(&eq_bm[c.x >> 5], 1u << (c.x & 31));
  }
}

constexpr int kBmThreads = 256;
constexpr int kBmWordsPerThread = 8;
constexpr int kBmWords = kBmThreads * kBmWordsPerThread;  // 2048 words = 65536 coordinates per block

__global__ void __launch_bounds__(kBmThreads) k_bm_count(const uint32_t* __restrict__ gt_bm,
                                                         const uint32_t* __restrict__ eq_bm, int64_t nbw,
                                                         uint32_t* blk_gt, uint32_t* blk_eq) {
  grid_begin();
  const int64_t w0 = (int64_t)blockIdx.x * kBmWords + (int64_t)threadIdx.x * kBmWordsPerThread;
  uint32_t gt = 0, eq = 0;
#pragma unroll
  for (int j = 0; j < kBmWordsPerThread; ++j) {
    if (w0 + j < nbw) {
      gt += __popc(__ldcg(&gt_bm[w0 + j]));
      eq += __popc(__ldcg(&eq_bm[w0 + j]));
    }
  }
  uint32_t tg, te;
  block_excl_scan(gt, &tg);
  block_excl_scan(eq, &te);
  if (threadIdx.x == 0) {
    blk_gt[blockIdx.x] = tg;
    blk_eq[blockIdx.x] = te;
  }
}

__global__ void __launch_bounds__(kScanThreads) k_scan(const uint32_t* __restrict__ blk_gt,
                                                       const uint32_t* __restrict__ blk_eq, int64_t nblk,
                                                       const SelectState* st, uint32_t* blk_base,
                                                       uint32_t* blk_eqx) {
  grid_begin();
  const uint32_t need_eq = __ldcg(&st->need_eq);
  uint32_t carry_gt = 0, carry_eq = 0;
  for (int64_t c0 = 0; c0 < nblk; c0 += blockDim.x) {
    const int64_t b = c0 + threadIdx.x;
    const uint32_t g = b < nblk ? blk_gt[b] : 0u;
    const uint32_t e = b < nblk ? blk_eq[b] : 0u;
    uint32_t tg, te;
    const uint32_t xg = block_excl_scan(g, &tg) + carry_gt;
    const uint32_t xe = block_excl_scan(e, &te) + carry_eq;
    if (b < nblk) {
      blk_base[b] = xg + (xe < need_eq ? xe : need_eq);
      blk_eqx[b] = xe;
    }
    carry_gt += tg;
    carry_eq += te;
  }
}

// Walks the set bits of each thread's words in index order: bits of gt_bm are taken, bits of
// eq_bm are taken while their rank among the keys equal to tau is below need_eq.
__global__ void __launch_bounds__(kBmThreads) k_bm_write(const uint32_t* __restrict__ gt_bm,
                                                         const uint32_t* __restrict__ eq_bm, int64_t nbw,
                                                         const SelectState* st, const uint32_t* __restrict__ blk_base,
                                                         const uint32_t* __restrict__ blk_eqx,
                                                         int64_t* __restrict__ idx_out, int64_t k) {
  grid_begin();
  const uint32_t need_eq = __ldcg(&st->need_eq);
  const uint32_t base = blk_base[blockIdx.x];
  const uint32_t eqx = blk_eqx[blockIdx.x];
  const int64_t w0 = (int64_t)blockIdx.x * kBmWords + (int64_t)threadIdx.x * kBmWordsPerThread;
  uint32_t g[kBmWordsPerThread], e[kBmWordsPerThread];
  uint32_t gt = 0, eq = 0;
#pragma unroll
  for (int j = 0; j < kBmWordsPerThread; ++j) {
    const bool in = w0 + j < nbw;
    g[j] = in ? __ldcg(&gt_bm[w0 + j]) : 0u;
    e[j] = in ? __ldcg(&eq_bm[w0 + j]) : 0u;
    gt += __popc(g[j]);
    eq += __popc(e[j]);
  }
  uint32_t tg, te;
  const uint32_t pre_gt = block_excl_scan(gt, &tg);
  const uint32_t pre_eq = block_excl_scan(eq, &te);
  if (gt + eq == 0) return;
  const uint32_t eq_quota = need_eq > eqx ? need_eq - eqx : 0u;  // this block's share of ties
  uint32_t pos = base + pre_gt + (pre_eq < eq_quota ? pre_eq : eq_quota);
  uint32_t eq_rank = pre_eq;
#pragma unroll
  for (int j = 0; j < kBmWordsPerThread; ++j) {
    uint32_t bits = g[j] | e[j];
    while (bits) {
      const int b = __ffs(bits) - 1;
      bits &= bits - 1u;
      bool take = (g[j] >> b) & 1u;
      if (!take) {
        take = eq_rank < eq_quota;
        ++eq_rank;
      }
      if (take) {
        if ((int64_t)pos < k) idx_out[pos] = (w0 + j) * 32 + b;
        ++pos;
      }
    }
  }
}

// ---- selection by one cluster ----------------------------------------------------------------
// For short vectors the selection's six kernels and their picks are almost all latency (33 us of a
// 92 us step at d = 2^20).  Here one cluster of 16 CTAs, the widest there is, does levels 2 and 3 and
// the ordered output in a single launch: each CTA owns a contiguous run of coordinates and keeps its
// bitmaps and candidates in shared memory; the histograms meet in the first CTA's shared memory, and
// cluster barriers stand where the kernels were.  Query and selection in us, k = d/1000 (d/100), six
// kernels / one cluster: d = 100k 35.2 / 22.0 (37.1 / 22.1), 300k 39.1 / 25.9 (42.4 / 28.2), 2^20 50.1 / 39.7
// (53.7 / 47.2), 2M 68.6 / 64.4 (72.2 / 75.7), 4M 108 / 112 (113 / 171): beyond 1.5 * 2^20 the 136 idle SMs
// cost more than the launches.  Writing many indices from 16 CTAs costs more than the launches as well,
// from about 819,200 coordinates on: k = d/50, d/10, d/2: d = 420k 40.9 / 32.1, 46.3 / 35.2, 59.5 / 43.0,
// 800k 49.4 / 45.7, 54.4 / 51.7, 68.1 / 65.3, 2^20 51.8 / 49.1, 57.9 / 58.4, 71.8 / 75.8, 1.5 * 2^20
// 58.7 / 62.4, 67.0 / 80.1, 79.2 / 104.  Keys that are all equal, which overflow the lists, follow the same
// line (k = d/10, 800k 98.6 / 92.4, 2^20 109 / 128).
constexpr int kSmallCtas = 16;
constexpr int kSmallThreads = 1024;
constexpr int kSmallList = 16384;                   // candidates kept per CTA
constexpr int64_t kSmallMaxDim = int64_t(3) << 19;  // 3072 bitmap words per CTA
constexpr int64_t kSmallAnyK = int64_t(25) << 15;   // up to this length for any k, beyond for k <= d/100

struct SmallShared {
  uint32_t h2[kBins];
  uint32_t h3[1 << kL3Bits];
  uint32_t sum[kBins];       // a histogram of the whole cluster
  uint2 list[kSmallList];    // candidates (index, key) of this CTA
  uint32_t n;                // how many there are (the list may hold fewer)
  uint32_t bin, rem;         // a pick
  uint32_t gt, eq;           // this CTA's keys above and equal to tau
};

// The bin of sum[0..nbins) that holds the k_rem-th largest key, and what is still to take in it.
__device__ __forceinline__ void pick_shared(SmallShared& sm, int nbins, uint32_t k_rem) {
  const int per = nbins / kSmallThreads;  // 1 or 2
  const int r0 = threadIdx.x * per;       // positions counted from the top bin
  uint32_t cnt[2] = {0u, 0u};
  for (int t = 0; t < per; ++t) cnt[t] = sm.sum[nbins - 1 - (r0 + t)];
  uint32_t total;
  uint32_t cum = block_excl_scan(cnt[0] + cnt[1], &total);
  for (int t = 0; t < per; ++t) {
    if (cum < k_rem && cum + cnt[t] >= k_rem) {
      sm.bin = (uint32_t)(nbins - 1 - (r0 + t));
      sm.rem = k_rem - cum;
    }
    cum += cnt[t];
  }
  __syncthreads();
}

// Calls f(index, key) for every coordinate of [c0, c1), c0 a multiple of 4.
template <typename F>
__device__ __forceinline__ void for_keys(const float* __restrict__ src, int64_t c0, int64_t c1, int vec, uint32_t kmask,
                                         const F& f) {
  for (int64_t b = c0; b < c1; b += 4 * kU * kSmallThreads) {
    float v[kU][4];
    int tm[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t i0 = b + 4 * ((int64_t)u * kSmallThreads + threadIdx.x);
      tm[u] = i0 < c1 ? (c1 - i0 < 4 ? (int)(c1 - i0) : 4) : 0;
      if (vec && tm[u] == 4) {
        const float4 x = __ldcg(reinterpret_cast<const float4*>(src + i0));
        v[u][0] = x.x; v[u][1] = x.y; v[u][2] = x.z; v[u][3] = x.w;
      } else {
#pragma unroll
        for (int t = 0; t < 4; ++t) v[u][t] = t < tm[u] ? __ldcg(src + i0 + t) : 0.f;
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int64_t i0 = b + 4 * ((int64_t)u * kSmallThreads + threadIdx.x);
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t < tm[u]) f((uint32_t)i0 + t, __float_as_uint(v[u][t]) & kmask);
    }
  }
}

// hist1: the level-1 histogram of the keys; every CTA picks its bin here.
__global__ void __cluster_dims__(kSmallCtas, 1, 1) __launch_bounds__(kSmallThreads, 1)
    k_select_small(const float* __restrict__ src, int64_t d, int vec, uint32_t kmask, const uint32_t* __restrict__ hist1,
                   uint32_t k, int64_t* __restrict__ idx_out) {
  grid_begin();
  extern __shared__ uint4 small_dyn[];
  SmallShared& sm = *reinterpret_cast<SmallShared*>(small_dyn);
  cg::cluster_group cluster = cg::this_cluster();
  const uint32_t rank = cluster.block_rank();
  const int64_t nbw = (d + 31) / 32;
  const int64_t per = (nbw + kSmallCtas - 1) / kSmallCtas;  // bitmap words of a CTA
  uint32_t* gt_bm = reinterpret_cast<uint32_t*>(small_dyn) + sizeof(SmallShared) / sizeof(uint32_t);
  uint32_t* eq_bm = gt_bm + per;
  const int64_t w0 = (int64_t)rank * per;
  const int nw = (int)(w0 >= nbw ? 0 : (nbw - w0 < per ? nbw - w0 : per));
  const int64_t c0 = w0 * 32, c1 = c0 + (int64_t)nw * 32 < d ? c0 + (int64_t)nw * 32 : d;

  for (int b = threadIdx.x; b < kBins; b += kSmallThreads) {
    sm.h2[b] = 0;
    sm.sum[b] = __ldcg(&hist1[b]);
  }
  for (int b = threadIdx.x; b < (1 << kL3Bits); b += kSmallThreads) sm.h3[b] = 0;
  for (int w = threadIdx.x; w < 2 * (int)per; w += kSmallThreads) gt_bm[w] = 0;  // both bitmaps
  if (threadIdx.x == 0) sm.n = 0;
  __syncthreads();
  pick_shared(sm, kBins, k);
  const uint32_t b1 = sm.bin, k1 = sm.rem;
  cluster.sync();  // every histogram is clear

  // level 2: keys above the bin are taken, those in it are candidates
  for_keys(src, c0, c1, vec, kmask, [&](uint32_t i, uint32_t key) {
    if ((key >> kL1Shift) < b1) return;
    if ((key >> kL1Shift) > b1) {
      const uint32_t at = i - (uint32_t)c0;
      atomicOr(&gt_bm[at >> 5], 1u << (at & 31));
      return;
    }
    atomicAdd(&sm.h2[(key >> kL2Shift) & (kBins - 1)], 1u);
    const uint32_t am = __activemask();
    const int lane = threadIdx.x & 31, leader = __ffs(am) - 1;
    uint32_t slot = 0;
    if (lane == leader) slot = atomicAdd(&sm.n, (uint32_t)__popc(am));
    slot = __shfl_sync(am, slot, leader) + __popc(am & ((1u << lane) - 1u));
    if (slot < (uint32_t)kSmallList) sm.list[slot] = make_uint2(i, key);
  });
  __syncthreads();
  const uint32_t n = sm.n;
  uint32_t* const total2 = cluster.map_shared_rank(sm.h2, 0);
  if (rank != 0)
    for (int b = threadIdx.x; b < kBins; b += kSmallThreads)
      if (sm.h2[b]) atomicAdd(&total2[b], sm.h2[b]);
  cluster.sync();
  for (int b = threadIdx.x; b < kBins; b += kSmallThreads) sm.sum[b] = total2[b];
  __syncthreads();
  pick_shared(sm, kBins, k1);
  const uint32_t p22 = (b1 << 11) | sm.bin, k2 = sm.rem;

  // level 3, over the candidates (the keys again where they overflow the list)
  const auto candidates = [&](const auto& f) {
    if (n <= (uint32_t)kSmallList) {
      for (uint32_t t = threadIdx.x; t < n; t += kSmallThreads) f(sm.list[t].x, sm.list[t].y);
    } else {
      for_keys(src, c0, c1, vec, kmask, [&](uint32_t i, uint32_t key) {
        if ((key >> kL1Shift) == b1) f(i, key);
      });
    }
  };
  candidates([&](uint32_t, uint32_t key) {
    if ((key >> kL2Shift) == p22) atomicAdd(&sm.h3[key & ((1u << kL3Bits) - 1u)], 1u);
  });
  __syncthreads();
  uint32_t* const total3 = cluster.map_shared_rank(sm.h3, 0);
  if (rank != 0)
    for (int b = threadIdx.x; b < (1 << kL3Bits); b += kSmallThreads)
      if (sm.h3[b]) atomicAdd(&total3[b], sm.h3[b]);
  cluster.sync();
  for (int b = threadIdx.x; b < (1 << kL3Bits); b += kSmallThreads) sm.sum[b] = total3[b];
  __syncthreads();
  pick_shared(sm, 1 << kL3Bits, k2);
  const uint32_t tau = (p22 << kL3Bits) | sm.bin, need_eq = sm.rem;

  candidates([&](uint32_t i, uint32_t key) {
    const uint32_t at = i - (uint32_t)c0;
    if (key > tau) atomicOr(&gt_bm[at >> 5], 1u << (at & 31));
    else if (key == tau) atomicOr(&eq_bm[at >> 5], 1u << (at & 31));
  });
  __syncthreads();

  // ordered output: this CTA's counts, those of the CTAs before it, then as in k_bm_write
  const int each = (nw + kSmallThreads - 1) / kSmallThreads;  // words of a thread
  const int t0 = threadIdx.x * each, t1 = t0 + each < nw ? t0 + each : nw;
  uint32_t gt = 0, eq = 0;
  for (int w = t0; w < t1; ++w) {
    gt += __popc(gt_bm[w]);
    eq += __popc(eq_bm[w]);
  }
  uint32_t all_gt, all_eq;
  const uint32_t pre_gt = block_excl_scan(gt, &all_gt), pre_eq = block_excl_scan(eq, &all_eq);
  if (threadIdx.x == 0) {
    sm.gt = all_gt;
    sm.eq = all_eq;
  }
  cluster.sync();
  uint32_t base = 0, eqx = 0;
  for (uint32_t c = 0; c < rank; ++c) {
    base += *cluster.map_shared_rank(&sm.gt, c);
    eqx += *cluster.map_shared_rank(&sm.eq, c);
  }
  base += eqx < need_eq ? eqx : need_eq;
  cluster.sync();  // no CTA leaves while others read its shared memory
  if (gt + eq == 0) return;
  const uint32_t eq_quota = need_eq > eqx ? need_eq - eqx : 0u;
  uint32_t pos = base + pre_gt + (pre_eq < eq_quota ? pre_eq : eq_quota);
  uint32_t eq_rank = pre_eq;
  for (int w = t0; w < t1; ++w) {
    uint32_t bits = gt_bm[w] | eq_bm[w];
    while (bits) {
      const int b = __ffs(bits) - 1;
      bits &= bits - 1u;
      bool take = (gt_bm[w] >> b) & 1u;
      if (!take) {
        take = eq_rank < eq_quota;
        ++eq_rank;
      }
      if (take) {
        if (pos < k) idx_out[pos] = c0 + (int64_t)w * 32 + b;
        ++pos;
      }
    }
  }
}

// ---- selection by full passes over est (fixed-scratch variant) -----------------------------

// Histogram of key bits [shift, shift + nbits) among keys whose bits above are the prefix
// picked at the previous level; ends with the pick of this level.
__global__ void __launch_bounds__(kBlock) k_hist(const float* __restrict__ est, int64_t d, int vec,
                                                 SelectState* st, uint32_t* hist, int shift, int nbits,
                                                 int level) {
  grid_begin();
  __shared__ uint32_t sh[kBins];
  const int nbins = 1 << nbits;
  for (int b = threadIdx.x; b < nbins; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const uint32_t prefix = __ldcg(&st->prefix);
  const int match_shift = shift + nbits;
  const int64_t nq = (d + 3) / 4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); q0 < nq; q0 += kU * stride) {
    float v[kU][4];
    int tm[kU];
    load_quads(est, d, vec, q0, stride, v, tm);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      uint32_t bins[4];
      bool any = false;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const uint32_t key = key_of(v[u][t]);
        const bool hit = t < tm[u] && (key >> match_shift) == prefix;
        bins[t] = hit ? ((key >> shift) & (uint32_t)(nbins - 1)) : kNone;
        any = any || hit;
      }
      if (__any_sync(kFull, any)) {  // most warps hold no key of the chosen bin
#pragma unroll
        for (int t = 0; t < 4; ++t) hist_add(sh, bins[t]);
      }
    }
  }
  hist_flush(sh, hist, nbins);
  last_block_pick(hist, nbits, st, level, 0);
}

// Segments of kSeg coordinates; a warp owns kWarpRun consecutive coordinates and reads them as
// kRows rows of 128 (lane l holds coordinates 4l .. 4l+3 of each row), so every load is a
// coalesced float4 and the ascending order of a warp's run is (row, lane, component).
constexpr int kSegThreads = 256;
constexpr int kSeg = 16384;
constexpr int kSegWarps = kSegThreads / 32;
constexpr int kWarpRun = kSeg / kSegWarps;   // 2048
constexpr int kRows = kWarpRun / 128;        // 16

template <bool VEC>
__device__ __forceinline__ void load_row(const float* __restrict__ est, int64_t i0, int64_t s1, float (&v)[4]) {
  if (VEC && i0 + 4 <= s1) {
    const float4 f = __ldg(reinterpret_cast<const float4*>(est + i0));
    v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
  } else {
#pragma unroll
    for (int t = 0; t < 4; ++t) v[t] = (i0 + t < s1) ? est[i0 + t] : 0.f;
  }
}

// Packed (eq << 16 | gt) counts of one segment; every field stays below 2^16.
__device__ __forceinline__ uint32_t count_key(uint32_t key, uint32_t tau) {
  return (key > tau ? 1u : 0u) | (key == tau ? (1u << 16) : 0u);
}

template <bool VEC>
__global__ void __launch_bounds__(kSegThreads) k_count(const float* __restrict__ est, int64_t d,
                                                       const SelectState* st, uint32_t* blk_gt,
                                                       uint32_t* blk_eq) {
  grid_begin();
  const uint32_t tau = __ldcg(&st->tau);
  const int64_t s0 = (int64_t)blockIdx.x * kSeg;
  const int64_t s1 = s0 + kSeg < d ? s0 + kSeg : d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t w0 = s0 + (int64_t)warp * kWarpRun;
  uint32_t cnt = 0;
  float v[kRows][4];
#pragma unroll
  for (int j = 0; j < kRows; ++j) load_row<VEC>(est, w0 + j * 128 + lane * 4, s1, v[j]);
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (w0 + j * 128 + lane * 4 + t < s1) cnt += count_key(key_of(v[j][t]), tau);
    }
  }
  uint32_t tot;
  block_excl_scan(cnt, &tot);
  if (threadIdx.x == 0) {
    blk_gt[blockIdx.x] = tot & 0xFFFFu;
    blk_eq[blockIdx.x] = tot >> 16;
  }
}

// Counts first (all rows in flight), then each row again from L1 to place its keys.
template <bool VEC>
__global__ void __launch_bounds__(kSegThreads) k_write(const float* __restrict__ est, int64_t d,
                                                       const SelectState* st, const uint32_t* __restrict__ blk_base,
                                                       const uint32_t* __restrict__ blk_eqx,
                                                       int64_t* __restrict__ idx_out, int64_t k) {
  grid_begin();
  __shared__ uint32_t warp_tot[kSegWarps];
  const uint32_t tau = __ldcg(&st->tau), need_eq = __ldcg(&st->need_eq);
  const int64_t s0 = (int64_t)blockIdx.x * kSeg;
  const int64_t s1 = s0 + kSeg < d ? s0 + kSeg : d;
  const uint32_t base = blk_base[blockIdx.x];
  const uint32_t eqx = blk_eqx[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t w0 = s0 + (int64_t)warp * kWarpRun;
  uint32_t cnt = 0;
  {
    float v[kRows][4];
#pragma unroll
    for (int j = 0; j < kRows; ++j) load_row<VEC>(est, w0 + j * 128 + lane * 4, s1, v[j]);
#pragma unroll
    for (int j = 0; j < kRows; ++j) {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (w0 + j * 128 + lane * 4 + t < s1) cnt += count_key(key_of(v[j][t]), tau);
      }
    }
  }
  // warp totals -> each warp's prefix inside the segment
  const uint32_t wsum = __shfl_sync(kFull, warp_incl_scan(cnt), 31);
  if (lane == 0) warp_tot[warp] = wsum;
  __syncthreads();
  uint32_t wpre = 0;
  for (int w = 0; w < warp; ++w) wpre += warp_tot[w];
  if (wsum == 0) return;
  uint32_t run = wpre;  // packed counts before the current row of this warp, within the segment
  const uint32_t eq_quota = need_eq > eqx ? need_eq - eqx : 0u;  // eq keys of this segment still taken
#pragma unroll 1
  for (int j = 0; j < kRows; ++j) {
    const int64_t i0 = w0 + j * 128 + lane * 4;
    float v[4];
    load_row<VEC>(est, i0, s1, v);
    uint32_t key[4];
    uint32_t c = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      key[t] = key_of(v[t]);
      if (i0 + t < s1) c += count_key(key[t], tau);
    }
    const uint32_t incl = warp_incl_scan(c);
    const uint32_t row_tot = __shfl_sync(kFull, incl, 31);
    if (c) {
      const uint32_t before = run + incl - c;
      const uint32_t gt_before = before & 0xFFFFu, eq_before = before >> 16;
      uint32_t pos = base + gt_before + (eq_before < eq_quota ? eq_before : eq_quota);
      uint32_t eq_rank = eq_before;  // rank among this segment's eq keys
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        if (i0 + t < s1) {
          bool take = key[t] > tau;
          if (key[t] == tau) {
            take = eq_rank < eq_quota;
            ++eq_rank;
          }
          if (take) {
            if ((int64_t)pos < k) idx_out[pos] = i0 + t;
            ++pos;
          }
        }
      }
    }
    run += row_tot;
  }
}

// ---- HEAVYMIX (Alg. 2 as printed) ----------------------------------------------------------

// Sum of squares of each row of the merged table in fp64; blockIdx.y is the row.
__global__ void __launch_bounds__(kBlock) k_row_sumsq(const float* __restrict__ T, uint32_t c, double* sumsq) {
  grid_begin();
  __shared__ double warp_acc[kBlock / 32];
  const int j = blockIdx.y;
  const float* row = T + (size_t)j * c;
  double acc = 0.0;
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < c; b += gridDim.x * blockDim.x) {
    const double v = (double)row[b];
    acc += v * v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o);
  if ((threadIdx.x & 31) == 0) warp_acc[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    double v = threadIdx.x < kBlock / 32 ? warp_acc[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    if (threadIdx.x == 0) atomicAdd(&sumsq[j], v);
  }
}

// l2sq = median over rows of the row sums of squares (the sketch's estimate of ||g||^2);
// theta = l2sq / k, the threshold of H.
// With `prune`, also the prune key of the query that follows: a coordinate with |est| < f,
// f^2 <= theta, lies outside H, and only its index enters the selection (through the random
// fill), so no repair is ever needed.
__global__ void k_heavy_theta(const double* __restrict__ sumsq, int r, int64_t k, double* theta,
                              double* l2sq_out, SelectState* st, int prune) {
  grid_begin();
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  double v[GS_MAX_ROWS];
  for (int j = 0; j < r; ++j) v[j] = __ldcg(&sumsq[j]);
  for (int a = 1; a < r; ++a) {
    const double t = v[a];
    int b = a - 1;
    while (b >= 0 && v[b] > t) {
      v[b + 1] = v[b];
      --b;
    }
    v[b + 1] = t;
  }
  const double m = (r & 1) ? v[r / 2] : 0.5 * (v[r / 2 - 1] + v[r / 2]);
  const double th = m / (double)k;
  theta[0] = th;
  if (l2sq_out) l2sq_out[0] = m;
  if (prune && th > 0.0 && th <= 1e300) {
    float f = __double2float_rd(sqrt(th));
    if ((double)f * (double)f > th) f = nextafterf(f, 0.f);  // the product is exact in double
    st->prune_key = key_of(f) & ~((1u << kL1Shift) - 1u);
  }
}

// ---- launchers -----------------------------------------------------------------------------

template <typename K>
int persistent_grid(K kernel, int64_t work_items, int block) {
  const int64_t need = (work_items + block - 1) / block;
  const int64_t cap = (int64_t)device_info().sms * blocks_per_sm((const void*)kernel, block);
  return (int)(need < 1 ? 1 : (need < cap ? need : cap));
}

template <int R>
cudaError_t launch_query_r(const QueryParams& p, cudaStream_t s) {
  auto kern = !is_pow2(p.c) ? k_query_mod<R> : p.keys ? k_query<R, true> : k_query<R, false>;
  if (p.keys) {
    // k_query_bits before it leaves an SM 28 KB of L1, in which few reads are in flight; a quarter of the SM's
    // memory shared holds the resident CTAs' histograms (d = 25.6M, r = 5, c = 2^18, k = 4 c: 944 -> 568 us)
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 25);
    if (e != cudaSuccess) return e;
  }
  launch(kern, persistent_grid(kern, (p.d + 3) / 4, kBlock), kBlock, s, p);
  return cudaGetLastError();
}

typedef cudaError_t (*QueryLauncher)(const QueryParams&, cudaStream_t);

template <int... Rs>
struct QueryTable {
  static constexpr QueryLauncher table[sizeof...(Rs)] = {&launch_query_r<Rs>...};
};
template <int... Rs>
constexpr QueryLauncher QueryTable<Rs...>::table[sizeof...(Rs)];

int bits_grid(int64_t d) {
  const int64_t need = ((d + 3) / 4 + kBitsBlock - 1) / kBitsBlock;
  return (int)(need < device_info().sms ? (need < 1 ? 1 : need) : device_info().sms);
}

// k_query_bits<R> for a pruning query whose first rows' classes fit kBitsBytes: the classes are
// written into `words` (f * c / 4 bytes of scratch) first.
template <typename... KArgs, typename... Args>
cudaError_t launch_on_every_sm(void (*kern)(KArgs...), int64_t d, size_t smem, cudaStream_t s, Args&&... args) {
  // the limit that every call sets: another thread's launch may stand between this call's setting and launch
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBitsBytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)bits_grid(d));
  cfg.blockDim = dim3(kBitsBlock);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int R>
cudaError_t launch_query_bits_r(const QueryParams& p, uint32_t* words, cudaStream_t s) {
  constexpr int kF = R / 2 + 1;
  const int64_t nwords = (int64_t)kF * (p.c / 32);  // words of one kind of bit
  const int64_t warps = (nwords + kBlock / 32 - 1) / (kBlock / 32), cap = (int64_t)device_info().sms * 8;
  launch(k_pbits, (int)(warps < cap ? warps : cap), kBlock, s, p.T, p.c, nwords, p.st, words);
  const size_t smem = (size_t)nwords * 2 * sizeof(uint32_t);
  GridSteps steps = {};
  for (int j = 0; j < kF; ++j) steps.a[j] = 8 * mulmod61(p.h.a[j], (uint64_t)bits_grid(p.d) * kBitsBlock * 4);
  auto kern = p.keys ? k_query_bits<R, true> : k_query_bits<R, false>;
  cudaError_t e = launch_on_every_sm(kern, p.d, smem, s, p, (const uint32_t*)words, steps);
  if (e == cudaSuccess && p.if_open && !p.keys)
    e = launch_on_every_sm(k_query_quads<R>, p.d, smem, s, p, (const uint32_t*)words);
  return e;
}

typedef cudaError_t (*BitsLauncher)(const QueryParams&, uint32_t*, cudaStream_t);

template <int... Rs>
struct BitsTable {
  static constexpr BitsLauncher table[sizeof...(Rs)] = {&launch_query_bits_r<Rs>...};
};
template <int... Rs>
constexpr BitsLauncher BitsTable<Rs...>::table[sizeof...(Rs)];

// Whether a pruning query of r rows and c (a power of two) columns classifies its first rows in
// shared memory.
bool query_uses_bits(int r, uint32_t c) {
  const uint64_t bytes = (uint64_t)(r / 2 + 1) * c / 4;
  return r >= 3 && r <= GS_MAX_ROWS && is_pow2(c) && c >= 64 && bytes <= kBitsBytes;
}

template <int R>
cudaError_t launch_repair_r(const QueryParams& p, uint32_t* hist_r, cudaStream_t s) {
  auto kern = k_repair<R>;
  // one CTA per SM: the kernel almost always returns at once, and a repair is rare
  launch(kern, device_info().sms, kBlock, s, p, hist_r);
  return cudaGetLastError();
}

typedef cudaError_t (*RepairLauncher)(const QueryParams&, uint32_t*, cudaStream_t);

template <int... Rs>
struct RepairTable {
  static constexpr RepairLauncher table[sizeof...(Rs)] = {&launch_repair_r<Rs>...};
};
template <int... Rs>
constexpr RepairLauncher RepairTable<Rs...>::table[sizeof...(Rs)];

template <int R>
cudaError_t launch_qsample_r(const QueryParams& p, uint32_t* hist_s, uint32_t j_target, cudaStream_t s) {
  auto kern = k_qsample<R>;
  const int64_t ns = ((p.d + 3) / 4 + kSampleQuads - 1) / kSampleQuads;
  launch(kern, persistent_grid(kern, ns, kBlock), kBlock, s, p, hist_s, j_target);
  return cudaGetLastError();
}

typedef cudaError_t (*SampleLauncher)(const QueryParams&, uint32_t*, uint32_t, cudaStream_t);

template <int... Rs>
struct SampleTable {
  static constexpr SampleLauncher table[sizeof...(Rs)] = {&launch_qsample_r<Rs>...};
};
template <int... Rs>
constexpr SampleLauncher SampleTable<Rs...>::table[sizeof...(Rs)];

// Rank, among the sampled keys, whose level-1 bin gives the prune key.  The sample holds n_s
// of the d coordinates; the number of them among the k - 1 keys above the k-th largest is
// at most hypergeometric with mean mu = k n_s / d.  Taking rank mu + 4 sqrt(mu) + 2 puts the
// sampled key below the k-th largest unless that count exceeds its mean by four standard
// deviations; for k below that rank it cannot exceed it at all.  0: no usable rank.
uint32_t sample_rank(int64_t d, int64_t k) {
  const int64_t ns = ((d + 3) / 4 + kSampleQuads - 1) / kSampleQuads;
  const int64_t last = (ns - 1) * kSampleQuads * 4;
  const int64_t n_s = 4 * (ns - 1) + (d - last < 4 ? d - last : 4);
  const double mu = (double)k * (double)n_s / (double)d;
  const double j = std::ceil(mu + 4.0 * std::sqrt(mu)) + 2.0;
  return j <= (double)n_s ? (uint32_t)j : 0u;
}

template <int R>
cudaError_t launch_gather_probe_r(const QueryParams& p, float* out, int64_t out_floats, cudaStream_t s) {
  auto kern = k_gather_probe<R>;
  const int grid = persistent_grid(k_query<R>, (p.d + 3) / 4, kBlock);  // the query's grid
  if (grid > out_floats) return cudaErrorInvalidValue;
  launch(kern, grid, kBlock, s, p, out);
  return cudaGetLastError();
}

typedef cudaError_t (*ProbeLauncher)(const QueryParams&, float*, int64_t, cudaStream_t);

template <int... Rs>
struct ProbeTable {
  static constexpr ProbeLauncher table[sizeof...(Rs)] = {&launch_gather_probe_r<Rs>...};
};
template <int... Rs>
constexpr ProbeLauncher ProbeTable<Rs...>::table[sizeof...(Rs)];

// Pruning applies on the fast path (c a power of two) with at least three rows, and from
// 2^22 coordinates up: below that the query takes a few tens of microseconds and the repair
// kernel's launch costs more than the skipped rows save (measured on the 2^20 workload).
constexpr int64_t kPruneMinDim = int64_t(1) << 22;
static_assert(kPruneMinDim > kSmallMaxDim, "a pruning query needs the level-1 pick, which the cluster does by itself");
bool can_prune(int r, uint32_t c, int64_t d) { return is_pow2(c) && r >= 3 && r <= GS_MAX_ROWS && d >= kPruneMinDim; }

template <int R>
cudaError_t launch_walk_r(const QueryParams& p, WalkParams& wk, cudaStream_t s) {
  const int64_t span = (int64_t)wk.outer * wk.outer_steps;
  wk.tiles = (wk.inner + kBlock - 1) / kBlock;
  const uint32_t blocks = wk.tiles * (uint32_t)((p.d + span - 1) / span);
  if (p.prune) launch(k_query_walk<R, true>, blocks, kBlock, s, p, wk);
  else launch(k_query_walk<R, false>, blocks, kBlock, s, p, wk);
  return cudaGetLastError();
}

typedef cudaError_t (*WalkLauncher)(const QueryParams&, WalkParams&, cudaStream_t);

template <int... Rs>
struct WalkTable {
  static constexpr WalkLauncher table[sizeof...(Rs)] = {&launch_walk_r<Rs>...};
};
template <int... Rs>
constexpr WalkLauncher WalkTable<Rs...>::table[sizeof...(Rs)];

// The walk pays where the reads it saves outweigh its steps.  Query with its selection in us, k_query /
// walk: all rows, r = 3, d = 4.2M, c = 2^16 79 / 85; r = 5, d = 2.1M, c = 2^16 72 / 73, d = 4.2M, c = 2^15
// 105 / 106, c = 2^17 113 / 104, d = 25.6M, c = 2^20 494 / 463; r = 9, d = 4.2M 177 / 165.  Pruning reads
// r/2 + 1 rows, so that two of them weigh more: r = 5, d = 25.6M, c = 2^20 395 / 342, r = 7, c = 2^18 510 / 444.
constexpr int64_t kWalkQueryMinDim = int64_t(1) << 22;
constexpr uint32_t kWalkQueryMinCols = 1u << 16;
// With a large k few coordinates settle in the first rows and nearly all of them are queued, which a pruning walk
// over a short vector does not repay: d = 4.2M, c = 2^18, k = d/30: r = 6 133 / 144, r = 8 177 / 197, r = 9 193 / 203
// (d = 25.6M: within 3 % of each other).
constexpr int64_t kWalkLargeKMinDim = int64_t(1) << 23;

// The walk of a query, or false where k_query serves it.
bool plan_walk(const QueryParams& p, const RowStrides& slow, WalkParams& wk) {
  if (slow.empty() || p.keys || p.r < (p.prune ? 3 : 5) || p.r > kWalkMaxRows || p.d < kWalkQueryMinDim || p.c < kWalkQueryMinCols)
    return false;
  if (p.prune && p.d < kWalkLargeKMinDim && p.k > p.d / 200) return false;
  const int nr = p.prune ? p.r / 2 + 1 : p.r;
  const int64_t max_steps = p.d / ((int64_t)device_info().sms * 1024 * 2);
  PairShape best;
  int first = 0, second = 1;
  for (int f = 0; f < 2; ++f) {  // either of the first two rows as the inner one
    const PairShape s = choose_pair(slow[f], slow[1 - f], p.d, kWalkSlots, max_steps < 64 ? max_steps : 64);
    if (s.changes < best.changes) {
      best = s;
      first = f;
      second = 1 - f;
    }
  }
  if (best.changes > 1.0) return false;
  std::memset(&wk, 0, sizeof(wk));
  wk.inner = (uint32_t)best.inner;
  wk.outer = (uint32_t)best.outer;
  wk.inner_steps = best.inner_steps;
  wk.outer_steps = best.outer_steps;
  for (int s = 0; s < nr; ++s) {
    const int j = s == 0 ? first : s == 1 ? second : s;
    WalkRow& r = wk.row[s];
    r.a8 = p.h8.a[j];
    r.b8 = p.h8.b[j];
    r.a28 = p.h8.a2[j];
    r.b28 = p.h8.b2[j];
    r.sa8 = 8 * mulmod61(p.h.a[j], (uint64_t)best.inner);
    r.sa28 = 8 * mulmod61(p.h.a2[j], (uint64_t)best.inner);
    for (int t = 0; t < 2; ++t) {
      // inner_steps - 1 inner strides are less than the outer one, and inner_steps >= 2
      const uint64_t jump = (uint64_t)(best.outer - (best.inner_steps - 1 - t) * best.inner);
      r.ja8[t] = 8 * mulmod61(p.h.a[j], jump);
      r.ja28[t] = 8 * mulmod61(p.h.a2[j], jump);
    }
    r.cells = p.T + (size_t)j * p.c;
  }
  return true;
}

cudaError_t launch_query(const QueryParams& p, const RowStrides& slow, cudaStream_t s) {
  WalkParams wk;
  if (plan_walk(p, slow, wk)) {
    using T = WalkTable<3, 4, 5, 6, 7, 8, 9>;
    return T::table[p.r - 3](p, wk, s);
  }
  using T = QueryTable<1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16>;
  return T::table[p.r - 1](p, s);
}

QueryParams make_query_params(const float* merged, const HashCoeffs& h, int r, uint32_t c, int64_t d,
                              int64_t k, float* est, uint32_t* hist, SelectState* st) {
  QueryParams qp;
  qp.T = merged;
  qp.est = est;
  qp.hist = hist;
  qp.st = st;
  qp.d = d;
  qp.k = (uint32_t)k;
  qp.r = r;
  qp.c = c;
  qp.cmask = c - 1;
  qp.cinv = bucket_inverse(c);
  qp.vec = (reinterpret_cast<uintptr_t>(est) & 15u) == 0 ? 1 : 0;
  qp.pick = 1;
  qp.prune = 0;
  qp.if_open = 0;
  qp.keys = nullptr;
  qp.theta = nullptr;
  qp.fill_seed = 0;
  qp.h = h;
  std::memset(&qp.h8, 0, sizeof(qp.h8));
  std::memset(qp.qa, 0, sizeof(qp.qa));
  for (int j = 0; j < r; ++j) {
    qp.h8.a[j] = 8 * h.a[j];
    qp.h8.b[j] = 8 * h.b[j];
    qp.h8.a2[j] = 8 * h.a2[j];
    qp.h8.b2[j] = 8 * h.b2[j];
    for (uint64_t t = 1; t <= 3 && j < GS_MAX_ROWS / 2 + 1; ++t) qp.qa[j][t - 1] = 8 * mulmod61(h.a[j], t);
  }
  return qp;
}

// Layout of the caller's workspace for the candidate pipeline.
struct Workspace {
  float* est;         // d
  uint32_t* hist;     // 5 * kBins: levels 1-3, level 1 again for k_repair, the sample's level 1
  SelectState* st;
  uint2* cand;        // d (index, key) pairs: room for every coordinate
  uint32_t* gt_bm;    // nbw words
  uint32_t* eq_bm;    // nbw words
  uint32_t* blk;      // 4 * nblk
  int64_t nbw, nblk;
};

Workspace carve(void* base, int64_t d) {
  Workspace w;
  char* p = static_cast<char*>(base);
  w.nbw = (d + 31) / 32;
  w.nblk = (w.nbw + kBmWords - 1) / kBmWords;
  w.est = reinterpret_cast<float*>(p);
  p += align256((size_t)d * sizeof(float));
  w.hist = reinterpret_cast<uint32_t*>(p);
  p += align256(5 * kBins * sizeof(uint32_t));
  w.st = reinterpret_cast<SelectState*>(p);
  p += align256(sizeof(SelectState));
  w.cand = reinterpret_cast<uint2*>(p);
  p += align256((size_t)d * sizeof(uint2));
  w.gt_bm = reinterpret_cast<uint32_t*>(p);
  p += align256((size_t)w.nbw * sizeof(uint32_t));
  w.eq_bm = reinterpret_cast<uint32_t*>(p);
  p += align256((size_t)w.nbw * sizeof(uint32_t));
  w.blk = reinterpret_cast<uint32_t*>(p);
  return w;
}

}  // namespace

size_t query_topk_workspace_bytes(int64_t d, int64_t k) {
  (void)k;
  const int64_t nbw = (d + 31) / 32;
  const int64_t nblk = (nbw + kBmWords - 1) / kBmWords;
  return align256((size_t)d * sizeof(float)) + align256(5 * kBins * sizeof(uint32_t)) +
         align256(sizeof(SelectState)) + align256((size_t)d * sizeof(uint2)) +
         2 * align256((size_t)nbw * sizeof(uint32_t)) + align256((size_t)nblk * 4 * sizeof(uint32_t));
}

namespace {

// Records marks[i] on s when the caller passed marks and set that entry (while a plan is captured).
cudaError_t mark(const cudaEvent_t* marks, int i, cudaStream_t s) {
  return (marks && marks[i]) ? cudaEventRecordWithFlags(marks[i], s, cudaEventRecordExternal) : cudaSuccess;
}

size_t small_smem(int64_t d) {
  const int64_t per = ((d + 31) / 32 + kSmallCtas - 1) / kSmallCtas;
  return sizeof(SmallShared) + 2 * (size_t)per * sizeof(uint32_t);
}

// Whether the current device can hold the cluster of k_select_small (asked once per device).  16 CTAs
// that take an SM each are twice the portable size: a partition of the device, or one with fewer SMs
// in use per processing cluster, may not place them, and short vectors are then selected by the kernels
// for long ones.
bool small_cluster_fits() {
  static std::mutex mu;
  static std::unordered_map<int, bool> fits;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::lock_guard<std::mutex> lock(mu);
  const auto it = fits.find(dev);
  if (it != fits.end()) return it->second;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kSmallCtas);
  cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = small_smem(kSmallMaxDim);
  int n = 0;
  cudaError_t e = cudaFuncSetAttribute(k_select_small, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_select_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k_select_small, &cfg);
  if (e != cudaSuccess) cudaGetLastError();  // not an error of this call
  return fits.emplace(dev, e == cudaSuccess && n > 0).first->second;
}

bool selects_small(int64_t d, int64_t k) {
  return d <= kSmallMaxDim && (d <= kSmallAnyK || k <= d / 100) && small_cluster_fits();
}

// Histograms and state (adjacent) and, unless the selection goes by one cluster, both bitmaps
// (adjacent) back to zero.
cudaError_t clear_selection(const Workspace& w, int64_t d, int64_t k, cudaStream_t s) {
  const size_t head = (size_t)(reinterpret_cast<char*>(w.st + 1) - reinterpret_cast<char*>(w.hist));
  cudaError_t err = cudaMemsetAsync(w.hist, 0, head, s);
  if (err == cudaSuccess && !selects_small(d, k))
    err = cudaMemsetAsync(w.gt_bm, 0, (size_t)(reinterpret_cast<char*>(w.blk) - reinterpret_cast<char*>(w.gt_bm)), s);
  return err;
}

// Whether k_query_quads is launched behind k_query_bits: were the cells noise alone, of standard deviation s, the
// medians would deviate by 1.25 s / sqrt(r), their k-th largest would be the quantile of that, and the share p of
// cells below it would follow.  Any structure in the vector raises the threshold and p; the prune key, a bin edge
// below a sample's rank, lowers them (r = 7, k = d/100: 0.31 by this, 0.52 found), hence the margin of 0.3.  What is
// not launched is not needed: k_query_bits then keeps the query whatever it finds.
bool may_stay_open(int r, int64_t d, int64_t k) {
  const double tail = (double)k / (double)d;
  double lo = 0.0, hi = 8.0;  // erfc(z) = tail
  for (int n = 0; n < 24; ++n) {
    const double z = 0.5 * (lo + hi);
    (std::erfc(z) > tail ? lo : hi) = z;
  }
  const double p = std::erf(lo * 1.2533 / std::sqrt((double)r));
  const int f = r / 2 + 1;
  const double few = std::pow(p, f - 1);
  return 1.0 - few * p - (f + 1 < r ? f * few * (1.0 - p) * p : 0.0) > kMostlyOpen - 0.3;
}

// The pruning query by k_query_bits; its words go in the candidate area, which the selection only
// uses after the query.
cudaError_t launch_query_bits(const QueryParams& p, const Workspace& w, cudaStream_t s) {
  using T = BitsTable<1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16>;
  return T::table[p.r - 1](p, reinterpret_cast<uint32_t*>(w.cand), s);
}

// The selection by one cluster, from the level-1 histogram on.
cudaError_t select_small(const float* src, int vec, uint32_t kmask, const uint32_t* hist1, int64_t d, int64_t k, int64_t* idx_out, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(k_select_small, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_select_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)small_smem(kSmallMaxDim));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kSmallCtas);
  cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = small_smem(d);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, k_select_small, src, d, vec, kmask, hist1, (uint32_t)k, idx_out);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// Levels 2 and 3 and the ordered output, after the level-1 histogram and pick of `src` keys.
cudaError_t select_from_keys(const Workspace& w, const float* src, int vec, uint32_t kmask, int64_t d, int64_t k,
                             int64_t* idx_out, cudaStream_t s) {
  launch(k_cand, persistent_grid(k_cand, (d + 3) / 4 / kU, kBlock), kBlock, s, src, d, vec, kmask, w.st,
                                                                                 w.hist + kBins, w.cand, w.gt_bm);
  const int small_grid = device_info().sms;
  launch(k_cand_hist3, small_grid, kBlock, s, w.cand, w.st, w.hist + 2 * kBins);
  launch(k_cand_mark, small_grid, kBlock, s, w.cand, w.st, w.gt_bm, w.eq_bm);
  uint32_t* blk_gt = w.blk;
  uint32_t* blk_eq = blk_gt + w.nblk;
  uint32_t* blk_base = blk_eq + w.nblk;
  uint32_t* blk_eqx = blk_base + w.nblk;
  const int nb = (int)w.nblk;
  launch(k_bm_count, nb, kBmThreads, s, w.gt_bm, w.eq_bm, w.nbw, blk_gt, blk_eq);
  launch(k_scan, 1, kScanThreads, s, blk_gt, blk_eq, w.nblk, w.st, blk_base, blk_eqx);
  launch(k_bm_write, nb, kBmThreads, s, w.gt_bm, w.eq_bm, w.nbw, w.st, blk_base, blk_eqx, idx_out, k);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_query_topk(const float* merged, const HashCoeffs& h, int r, uint32_t c,
                              int64_t d, int64_t k, int64_t* idx_out, float* est_out,
                              void* workspace, cudaStream_t s, const RowStrides& slow, const cudaEvent_t* marks) {
  Workspace w = carve(workspace, d);
  float* est = est_out ? est_out : w.est;
  cudaError_t err = clear_selection(w, d, k, s);
  if (err != cudaSuccess) return err;
  if ((err = mark(marks, 0, s)) != cudaSuccess) return err;

  QueryParams qp = make_query_params(merged, h, r, c, d, k, est, w.hist, w.st);
  // rows are pruned only while the estimate stays internal: a caller's est_out gets every value
  const uint32_t j_target = sample_rank(d, k);
  qp.prune = (!est_out && can_prune(r, c, d) && j_target > 0) ? 1 : 0;
  qp.pick = selects_small(d, k) ? 0 : 1;
  if (qp.prune) {
    using T = SampleTable<1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16>;
    if ((err = T::table[r - 1](qp, w.hist + 4 * kBins, j_target, s)) != cudaSuccess) return err;
  }
  if (qp.prune && query_uses_bits(r, c)) {
    qp.if_open = may_stay_open(r, d, k) ? 1 : 0;
    if ((err = launch_query_bits(qp, w, s)) != cudaSuccess) return err;
  } else if ((err = launch_query(qp, slow, s)) != cudaSuccess) {
    return err;
  }
  if (qp.prune) {
    using T = RepairTable<1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16>;
    if ((err = T::table[r - 1](qp, w.hist + 3 * kBins, s)) != cudaSuccess) return err;
  }
  if ((err = mark(marks, 1, s)) != cudaSuccess) return err;
  if (selects_small(d, k)) err = select_small(est, qp.vec, 0x7FFFFFFFu, w.hist, d, k, idx_out, s);
  else err = select_from_keys(w, est, qp.vec, 0x7FFFFFFFu, d, k, idx_out, s);
  return err != cudaSuccess ? err : mark(marks, 2, s);
}

cudaError_t launch_query_ceiling_probe(const float* merged, const HashCoeffs& h, int r, uint32_t c, int64_t d,
                                       float* out, int64_t out_floats, cudaStream_t s) {
  if (!is_pow2(c) || r < 1 || r > GS_MAX_ROWS) return cudaErrorInvalidValue;
  const QueryParams qp = make_query_params(merged, h, r, c, d, 1, nullptr, nullptr, nullptr);
  using T = ProbeTable<1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 12, 13, 14, 15, 16>;
  return T::table[r - 1](qp, out, out_floats, s);
}

size_t heavymix_workspace_bytes(int64_t d, int64_t k) {
  return query_topk_workspace_bytes(d, k) + align256((size_t)d * sizeof(uint32_t)) + 256;
}

cudaError_t launch_query_heavymix(const float* merged, const HashCoeffs& h, int r, uint32_t c, int64_t d,
                                  int64_t k, uint64_t fill_seed, int64_t* idx_out, float* est_out, double* l2sq_out,
                                  void* workspace, cudaStream_t s, const cudaEvent_t* marks) {
  Workspace w = carve(workspace, d);
  char* extra = static_cast<char*>(workspace) + query_topk_workspace_bytes(d, k);
  uint32_t* keys = reinterpret_cast<uint32_t*>(extra);
  double* sumsq = reinterpret_cast<double*>(extra + align256((size_t)d * sizeof(uint32_t)));
  double* theta = sumsq + GS_MAX_ROWS;
  float* est = est_out ? est_out : w.est;
  cudaError_t err = clear_selection(w, d, k, s);
  if (err == cudaSuccess) err = cudaMemsetAsync(sumsq, 0, 256, s);
  if (err == cudaSuccess) err = mark(marks, 0, s);
  if (err != cudaSuccess) return err;

  // the threshold first (it reads only the table), so that the query can skip rows below it
  const int gx = (int)(((int64_t)c + kBlock - 1) / kBlock < 4 * device_info().sms ? ((int64_t)c + kBlock - 1) / kBlock
                                                                                  : 4 * device_info().sms);
  launch(k_row_sumsq, dim3(gx, r), kBlock, s, merged, c, sumsq);
  const int prune = (!est_out && can_prune(r, c, d)) ? 1 : 0;
  launch(k_heavy_theta, 1, 32, s, sumsq, r, k, theta, l2sq_out, w.st, prune);
  // the query stores each coordinate's composite key and picks on their level-1 histogram
  QueryParams qp = make_query_params(merged, h, r, c, d, k, est, w.hist, w.st);
  qp.prune = prune;
  qp.pick = selects_small(d, k) ? 0 : 1;
  qp.keys = keys;
  qp.theta = theta;
  qp.fill_seed = fill_seed;
  // The classified query first, where the classes fit; k_query where they do not, or where that query finds too
  // few coordinates settled (its CTAs return at once otherwise).  Query with its selection in us, classified /
  // k_query, d = 25.6M, r = 5, c = 2^18, k = 0.3 c, 0.6 c, c, 4 c: 239 / 454, 379 / 483, 483 / 491, 890 / 560.
  // A row of squared norm l2sq has at most k cells that reach l2sq / k, and k / 0.76 that reach the bin edge
  // below it: with k <= c / 8 five cells in six are inside, enough for any r, and k_query is not launched (the
  // classified query then keeps the whole of it, also where the rows' norms differ widely).
  const bool bits = prune && query_uses_bits(r, c);
  qp.if_open = bits && k > (int64_t)c / 8 && heavy_open(r) < 1.f ? 1 : 0;
  if (bits) err = launch_query_bits(qp, w, s);
  if (err == cudaSuccess && (!bits || qp.if_open)) err = launch_query(qp, RowStrides(), s);
  if (err != cudaSuccess) return err;
  if ((err = mark(marks, 1, s)) != cudaSuccess) return err;
  const float* src = reinterpret_cast<const float*>(keys);
  if (selects_small(d, k)) err = select_small(src, 1, 0xFFFFFFFFu, w.hist, d, k, idx_out, s);
  else err = select_from_keys(w, src, 1, 0xFFFFFFFFu, d, k, idx_out, s);
  return err != cudaSuccess ? err : mark(marks, 2, s);
}

// ---- scratch without allocation ---------------------------------------------------------
// For callers that cannot allocate: the selection scratch of the query (three histograms,
// the state, and four counters per segment of kSeg coordinates, enough for d up to
// GS_NOALLOC_MAX_DIM) lives in one array of the library's device memory.
namespace {

constexpr int64_t kNoallocMaxSegs = (GS_NOALLOC_MAX_DIM + kSeg - 1) / kSeg;
constexpr size_t kNoallocHistBytes = 3 * kBins * sizeof(uint32_t);   // multiple of 256
constexpr size_t kNoallocStateBytes = 256;
constexpr size_t kNoallocScratchBytes =
    kNoallocHistBytes + kNoallocStateBytes + (size_t)kNoallocMaxSegs * 4 * sizeof(uint32_t);
static_assert(sizeof(SelectState) <= kNoallocStateBytes, "state slot too small");

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocScratchBytes];

// Unique id of the context current on this thread (0 when none is current or the driver's
// entry points are unavailable).  A device reset or a rebuilt primary context gets a new id
// and a new load of this library's module, hence a new address of g_noalloc_scratch.  The
// two driver calls are reached through the runtime's entry-point query, so the library does
// not link the driver library itself.
unsigned long long current_context_id() {
  typedef CUresult (*GetCurrent)(CUcontext*);
  typedef CUresult (*GetId)(CUcontext, unsigned long long*);
  static GetCurrent get_current = nullptr;
  static GetId get_id = nullptr;
  static bool looked_up = false;
  if (!looked_up) {
    looked_up = true;
    void* f1 = nullptr;
    void* f2 = nullptr;
    cudaDriverEntryPointQueryResult q1, q2;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f1, 12000, cudaEnableDefault, &q1) == cudaSuccess &&
        cudaGetDriverEntryPointByVersion("cuCtxGetId", &f2, 12000, cudaEnableDefault, &q2) == cudaSuccess &&
        q1 == cudaDriverEntryPointSuccess && q2 == cudaDriverEntryPointSuccess) {
      get_current = reinterpret_cast<GetCurrent>(f1);
      get_id = reinterpret_cast<GetId>(f2);
    }
    cudaGetLastError();
  }
  if (!get_current || !get_id) return 0;
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (get_current(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, &id) != CUDA_SUCCESS) return 0;
  return id;
}

// Device address of g_noalloc_scratch on the current device.  It is looked up once per
// device and context (cudaGetSymbolAddress, a host-side query that allocates nothing) and
// cached under the context's id, so a reset device gets a fresh lookup.  Without a readable
// id the lookup runs on every call.
cudaError_t noalloc_scratch(void** out) {
  struct Entry {
    unsigned long long ctx;
    void* addr;
  };
  static std::mutex mu;
  static Entry cache[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  unsigned long long ctx = current_context_id();
  if (ctx != 0 && cache[dev].ctx == ctx && cache[dev].addr) {
    *out = cache[dev].addr;
    return cudaSuccess;
  }
  void* p = nullptr;
  e = cudaGetSymbolAddress(&p, g_noalloc_scratch);  // also makes the device's context current
  if (e != cudaSuccess) return e;
  if (ctx == 0) ctx = current_context_id();
  cache[dev].ctx = ctx;
  cache[dev].addr = ctx ? p : nullptr;
  *out = p;
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_query_topk_noalloc(const float* merged, const HashCoeffs& h, int r, uint32_t c,
                                      int64_t d, int64_t k, int64_t* idx_out, float* est_out,
                                      cudaStream_t s, const RowStrides& slow) {
  if (d > GS_NOALLOC_MAX_DIM || est_out == nullptr) return cudaErrorInvalidValue;
  void* base = nullptr;
  cudaError_t err = noalloc_scratch(&base);
  if (err != cudaSuccess) return err;
  char* p = static_cast<char*>(base);
  uint32_t* hist = reinterpret_cast<uint32_t*>(p);
  SelectState* st = reinterpret_cast<SelectState*>(p + kNoallocHistBytes);
  const int64_t nseg = (d + kSeg - 1) / kSeg;
  uint32_t* blk_gt = reinterpret_cast<uint32_t*>(p + kNoallocHistBytes + kNoallocStateBytes);
  uint32_t* blk_eq = blk_gt + nseg;
  uint32_t* blk_base = blk_eq + nseg;
  uint32_t* blk_eqx = blk_base + nseg;
  // the histograms and the state must start at zero; the segment counters are overwritten
  err = cudaMemsetAsync(hist, 0, kNoallocHistBytes + kNoallocStateBytes, s);
  if (err != cudaSuccess) return err;

  QueryParams qp = make_query_params(merged, h, r, c, d, k, est_out, hist, st);
  qp.pick = selects_small(d, k) ? 0 : 1;
  if ((err = launch_query(qp, slow, s)) != cudaSuccess) return err;
  if (selects_small(d, k)) return select_small(est_out, qp.vec, 0x7FFFFFFFu, hist, d, k, idx_out, s);
  const int hgrid = persistent_grid(k_hist, (d + 3) / 4 / kU, kBlock);
  launch(k_hist, hgrid, kBlock, s, est_out, d, qp.vec, st, hist + kBins, kL2Shift, 11, 1);
  launch(k_hist, hgrid, kBlock, s, est_out, d, qp.vec, st, hist + 2 * kBins, 0, kL3Bits, 2);
  const int nb = (int)nseg;
  if (qp.vec) launch(k_count<true>, nb, kSegThreads, s, est_out, d, st, blk_gt, blk_eq);
  else launch(k_count<false>, nb, kSegThreads, s, est_out, d, st, blk_gt, blk_eq);
  launch(k_scan, 1, kScanThreads, s, blk_gt, blk_eq, nseg, st, blk_base, blk_eqx);
  if (qp.vec) launch(k_write<true>, nb, kSegThreads, s, est_out, d, st, blk_base, blk_eqx, idx_out, k);
  else launch(k_write<false>, nb, kSegThreads, s, est_out, d, st, blk_base, blk_eqx, idx_out, k);
  return cudaGetLastError();
}

}  // namespace gs
