// Internal declarations shared by the translation units of the gs-SGD compression library.
// Device-side Count Sketch hashing over the Mersenne prime 2^61 - 1, kernel parameter
// blocks and the host-side launcher entry points called by the C ABI in gs_api.cu.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "gs_sketch.h"

#include <utility>
#include <vector>

namespace gs {

constexpr uint64_t kP61 = (1ull << 61) - 1;
constexpr int kMaxGroup = 16;       // widest worker group interleaved in one table
constexpr int kBlock = 256;         // threads per CTA for the streaming kernels

// Hash coefficients of every row: h_j uses (a[j], b[j]); s_j uses (a2[j], b2[j]).
struct HashCoeffs {
  uint64_t a[GS_MAX_ROWS], b[GS_MAX_ROWS], a2[GS_MAX_ROWS], b2[GS_MAX_ROWS];
};

// ---- Mersenne-prime arithmetic ----------------------------------------------------------
// x mod p is congruent to (x & p) + (x >> 61) because 2^61 = 1 (mod p).
__device__ __forceinline__ uint64_t fold61(uint64_t x) { return (x & kP61) + (x >> 61); }

// (a*i + b) mod p for a, b < p and i < 2^32.  a is split into 32-bit halves:
//   a*i = ahi*i*2^32 + alo*i,  and  ahi*i*2^32 = q*2^61 + rem*2^32 = q + rem*2^32 (mod p)
// with q = (ahi*i) >> 29 and rem = (ahi*i) mod 2^29.  Every partial sum stays below 2^63.
__device__ __forceinline__ uint64_t affine61(uint64_t a, uint64_t b, uint32_t i) {
  const uint64_t p0 = (uint64_t)(uint32_t)a * i;          // < 2^64
  const uint64_t p1 = (uint64_t)(uint32_t)(a >> 32) * i;  // < 2^61
  uint64_t s = (p1 >> 29) + ((p1 & ((1ull << 29) - 1)) << 32) + fold61(p0) + b;
  s = fold61(s);                                          // < p + 4
  return s >= kP61 ? s - kP61 : s;
}

// x + a mod p for x, a < p: the next coordinate's hash value in the incremental form
// (a*(i+1) + b) = (a*i + b) + a.
__device__ __forceinline__ uint64_t step61(uint64_t x, uint64_t a) {
  x += a;
  return x >= kP61 ? x - kP61 : x;
}

// ---- the same by carries ------------------------------------------------------------------
// For the kernels that are bound by their integer instructions (k_query_bits, k_insert_chain; k_query,
// which is bound by its reads, took 4 % longer with it).  A hash value x in [0, p),
// p = 2^61 - 1, is held as Y = 8 (x + 1), which lies in [8, 2^64 - 8].  For a residue s the 64-bit sum
// Y + 8 s = 8 (x + s + 1) overflows exactly when x + s >= p, and then (x + s) mod p is represented by
// the wrapped sum plus 8, since 8 p = 2^64 - 8.  So an addition and its carry-out reduce exactly,
// without a compare, and the low word of Y alone gives the bucket and the sign.
struct Rot {
  uint32_t lo, hi;
};

// The representation of (x + s) mod p from that of x; s8 = 8 s, s in [0, p).
__device__ __forceinline__ Rot rot_add(Rot y, uint64_t s8) {
  uint32_t lo, hi, carry;
  asm("add.cc.u32 %0, %3, %5;\n\taddc.cc.u32 %1, %4, %6;\n\taddc.u32 %2, 0, 0;"
      : "=r"(lo), "=r"(hi), "=r"(carry)
      : "r"(y.lo), "r"(y.hi), "r"((uint32_t)s8), "r"((uint32_t)(s8 >> 32)));
  Rot out;
  asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, 0;" : "=r"(out.lo), "=r"(out.hi) : "r"(lo), "r"(hi), "r"(8u * carry));
  return out;
}

// The low word of rot_add.
__device__ __forceinline__ uint32_t rot_add_lo(Rot y, uint64_t s8) {
  uint32_t lo, carry;
  asm("{\n\t.reg .u32 hi;\n\tadd.cc.u32 %0, %2, %4;\n\taddc.cc.u32 hi, %3, %5;\n\taddc.u32 %1, 0, 0;\n\t}"
      : "=r"(lo), "=r"(carry)
      : "r"(y.lo), "r"(y.hi), "r"((uint32_t)s8), "r"((uint32_t)(s8 >> 32)));
  return lo + 8u * carry;
}

// The representation of a i mod p, from a8 = 8 a, for i < 2^32: 8 a i = h 2^64 + l with h < 2^32, and
// 2^64 is 8 modulo 2^64 - 8, so l + 8 h + 8 with its carry folded in as above (l / 8 + h < 2 p).
__device__ __forceinline__ Rot rot_mul(uint64_t a8, uint32_t i) {
  const uint64_t w = (uint64_t)(uint32_t)a8 * i;
  const uint64_t z = (uint64_t)(uint32_t)(a8 >> 32) * i + (w >> 32);
  return rot_add(Rot{(uint32_t)w, (uint32_t)z}, 8ull * (uint32_t)(z >> 32) + 8ull);
}

// The representation of (a i + b) mod p, and its low word.
__device__ __forceinline__ Rot rot_at(uint64_t a8, uint64_t b8, uint32_t i) { return rot_add(rot_mul(a8, i), b8); }
__device__ __forceinline__ uint32_t rot_at_lo(uint64_t a8, uint64_t b8, uint32_t i) {
  return rot_add_lo(rot_mul(a8, i), b8);
}

// From the low word: the bucket for c a power of two, and the sign bit (bit 31 set when x is odd).
__device__ __forceinline__ uint32_t rot_bucket(uint32_t lo, uint32_t cmask) { return ((lo >> 3) - 1u) & cmask; }
__device__ __forceinline__ uint32_t rot_signbit(uint32_t lo) { return (~lo & 8u) << 28; }

// x mod c.  For c not a power of two, with cinv = floor(2^64 / c): the estimate x * cinv >> 64 of the
// quotient is at most 1 below it (x < 2^61), so the remainder needs one correction.
template <bool POW2>
__device__ __forceinline__ uint32_t bucket_of(uint64_t x, uint32_t c, uint32_t cmask, uint64_t cinv) {
  if (POW2) return (uint32_t)x & cmask;
  const uint32_t r = (uint32_t)x - (uint32_t)__umul64hi(x, cinv) * c;
  return r >= c ? r - c : r;
}

// Sign bit (bit 31 set for s = -1): s_j(i) = -1 when the second hash value is odd.
__device__ __forceinline__ uint32_t signbit_of(uint64_t y) { return ((uint32_t)y & 1u) << 31; }

__device__ __forceinline__ float apply_sign(float v, uint32_t sbit) {
  return __uint_as_float(__float_as_uint(v) ^ sbit);
}

// ---- fp32 reductions into L2-resident tables -------------------------------------------
__device__ __forceinline__ void red_add_f32(float* p, float v) {
  asm volatile("red.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}
__device__ __forceinline__ void red_add_v2(float* p, float v0, float v1) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(v0), "f"(v1) : "memory");
}
__device__ __forceinline__ void red_add_v4(float* p, float v0, float v1, float v2, float v3) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v0), "f"(v1),
               "f"(v2), "f"(v3)
               : "memory");
}

// ---- L2 eviction priorities -------------------------------------------------------------
// Cache policies for the insert.  The sketch table receives every reduction and should stay in L2:
// evict_last in every kernel.  Vector streams: normal in k_accumulate_chain; in k_insert_chain, which
// only reads them, evict_first once the vectors no longer fit L2 from one row to the next
// (ChainParams::resident); in the insert by reductions evict_first only where the table needs several
// passes (InsertParams::evict; 64 MiB row slices and 8 workers' streams, every row by reductions: five row
// passes 21.9 ms with both policies, 25.0 without).  Streams that are written must not carry it lightly: a
// line that two warps share, as every line of a vector that does not start on a 128-byte boundary does, may
// be evicted half written.  Accumulating 8 vectors of 25,557,032, 32 bytes off such a boundary: 0.645 ms
// without the mark, 0.745 with it.
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ uint64_t policy_normal() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ float ld_hinted(const float* p, uint64_t pol) {
  float v;
  asm volatile("ld.global.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ float4 ld_hinted4(const float* p, uint64_t pol) {
  float4 v;
  asm volatile("ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ float4 ld_stream(const float* p, uint64_t pol) {
  float4 v;
  asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ void st_stream(float* p, float4 v, uint64_t pol) {
  asm volatile("st.global.L1::no_allocate.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "f"(v.x),
               "f"(v.y), "f"(v.z), "f"(v.w), "l"(pol)
               : "memory");
}
__device__ __forceinline__ void red_add_v4_keep(float* p, float v0, float v1, float v2, float v3, uint64_t pol) {
  asm volatile("red.global.add.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "f"(v0), "f"(v1),
               "f"(v2), "f"(v3), "l"(pol)
               : "memory");
}

// ---- parameter blocks --------------------------------------------------------------------
struct InsertParams {
  float* u[kMaxGroup];
  float* e[kMaxGroup];
  const float* g[kMaxGroup];
  float* table;      // base of the group's interleaved table [r][c][W]
  int64_t d;
  int32_t nw;        // lanes of the group carrying a worker in this call
  int32_t lane;      // single-vector insert: the lane written
  int32_t r;
  int32_t j0, j1;    // rows inserted by this launch: [j0, j1)
  uint32_t c, cmask;
  uint64_t cinv;     // bucket_inverse(c)
  float rho;
  int32_t evict;     // the table does not fit L2 beside the streams: mark these evict_first
  int64_t winmask;   // request-ceiling probe only: vector offsets are taken modulo winmask + 1
  HashCoeffs h;
};

// Rows inserted by chains of coordinates (k_insert_chain), in launch order.
struct ChainRow {
  uint64_t a8, b8, a28, b28;  // 8 times the row's hash coefficients
  uint64_t sa8, sa28;         // 8 (a * stride mod p), 8 (a2 * stride mod p): one step along a chain
  float* cells;           // the row's cells, ChainParams::pitch floats apart
  int64_t stride;         // coordinates between two steps of a chain
  int32_t steps;          // coordinates of a chain
  uint32_t tiles;         // CTAs across the stride
  uint32_t first_block;   // first CTA of this row
};

// How k_accumulate_chain walks the coordinates: chains of `steps` quads, `stride` quads apart.
struct QuadWalk {
  int64_t stride;
  int32_t steps;
  uint32_t tiles;  // CTAs across the stride
};

struct ChainParams {
  const float* e[kMaxGroup];
  int64_t d;
  uint32_t cmask;
  int32_t nw;             // vectors inserted
  int32_t pitch;          // floats between two cells of a row
  int32_t nrows;
  int32_t resident;       // the vectors fit L2 between two rows
  ChainRow row[GS_MAX_ROWS];
};

struct Convergent;
typedef std::vector<std::vector<Convergent>> RowStrides;  // per row, see slow_strides

struct MergeParams {
  const float* tables;   // all groups, [group][r][c][W]
  float* merged;         // [r][c]
  int64_t cells;         // r*c
  int64_t group_stride;  // r*c*W floats
  int32_t P;
};

struct MergeListParams {
  const float* tables[GS_MAX_WORKERS];   // worker 0's table of each sketch, [r][c][lane_stride]
  int32_t lane_stride[GS_MAX_WORKERS];
  float* merged;                          // [r][c]
  int64_t cells;
  int32_t P;
};

struct GatherParams {
  float* u[GS_MAX_WORKERS];
  float* e[GS_MAX_WORKERS];
  const int64_t* idx;
  float* vals;
  float* w;          // weights to update with the gathered values (nullable)
  float lr;
  int64_t k, d;
  int32_t P;
};

// ---- launchers (return a cudaError_t from the launch) ------------------------------------
struct DeviceInfo {
  int sms;
};
DeviceInfo device_info();
// Resident CTAs per SM for `kernel` at `block` threads (cached per kernel address).
int blocks_per_sm(const void* kernel, int block);

cudaError_t launch_accumulate(float* u, float* e, const float* g, int64_t d, float rho,
                              cudaStream_t s);
// acc: accumulate (read g, u, e; write u, e) before inserting; otherwise insert e as it is.
cudaError_t launch_accumulate_insert(const InsertParams& p, int W, bool acc, bool vec, cudaStream_t s);
// The accumulate pass with rows [p.j0, p.j1) inserted (at least one; c a power of two), walking the
// chains of `wk` (tiles filled in here), along which row p.j0 keeps its buckets.
cudaError_t launch_accumulate_chain(const InsertParams& p, QuadWalk wk, int W, bool vec, cudaStream_t s);
cudaError_t launch_insert_lane(const InsertParams& p, int W, cudaStream_t s);
// Inserts the vectors p.e[0..nw) into the p.nrows rows of p.row (c a power of two; the strides and
// steps chosen by the caller, tiles and first_block filled in here).  W in {1, 2, 4, 8, 16}: workers
// per cell written; p.pitch == W unless W == 1.
cudaError_t launch_insert_chain(ChainParams& p, int W, cudaStream_t s);
// The fused insert's instruction stream with every vector access at offset i & p.winmask (the
// vectors are windows of winmask + 1 floats, 16-byte aligned): the same loads, stores and
// cell reductions, with the streams held in L2.  W in {4, 8, 16}, c a power of two.
cudaError_t launch_insert_ceiling_probe(const InsertParams& p, int W, bool acc, cudaStream_t s);
// Shared-memory-staged insert of the (already accumulated) vectors p.e[0..nw) into rows
// [j0, j1) of a W-wide group table; needs a tile of c * wt * 4 bytes (staged_tile_width).
constexpr size_t kStagedSmemBytes = size_t(200) << 10;
int staged_tile_width(uint32_t c, int W);   // workers per tile, 0 when no tile fits
cudaError_t launch_insert_staged(const InsertParams& p, int W, cudaStream_t s);
cudaError_t launch_hash_eval(const HashCoeffs& h, int r, uint32_t c, const int64_t* coords,
                             int64_t n, int32_t* bucket_out, int8_t* sign_out, cudaStream_t s);
cudaError_t launch_merge(const MergeParams& p, int W, cudaStream_t s);
cudaError_t launch_merge_list(const MergeListParams& p, cudaStream_t s);
cudaError_t launch_gather_and_zero(const GatherParams& p, cudaStream_t s);
cudaError_t launch_apply_update(float* w, int64_t d, const int64_t* idx, const float* vals, int64_t k, float lr,
                                cudaStream_t s);

size_t query_topk_workspace_bytes(int64_t d, int64_t k);

// momentum and error kept as sketches
cudaError_t launch_query_at(const float* T, const HashCoeffs& h, int r, uint32_t c, const int64_t* idx, int64_t k,
                            float* out, cudaStream_t s);
cudaError_t launch_add_sparse(float* T, const HashCoeffs& h, int r, uint32_t c, const int64_t* idx, const float* vals,
                              int64_t k, float scale, cudaStream_t s);
cudaError_t launch_take(const float* src, int64_t n, const int64_t* idx, int64_t k, float* out, cudaStream_t s);
// slow: the slow strides of the first two rows (empty unless c is a power of two and r >= 3).
// marks (nullable): three events recorded, when set, before the query, between the query
// (sample, median query, repair check) and the selection, and after the selection.
cudaError_t launch_query_topk(const float* merged, const HashCoeffs& h, int r, uint32_t c,
                              int64_t d, int64_t k, int64_t* idx_out, float* est_out,
                              void* workspace, cudaStream_t s, const RowStrides& slow,
                              const cudaEvent_t* marks = nullptr);
// Request-ceiling probe of the median query: its loads (all r rows) without median, store or
// histogram; out receives one float per CTA (out_floats must cover the grid).  c a power of two.
cudaError_t launch_query_ceiling_probe(const float* merged, const HashCoeffs& h, int r, uint32_t c, int64_t d,
                                       float* out, int64_t out_floats, cudaStream_t s);
// HEAVYMIX selection (Alg. 2 as printed) from the merged table; l2sq_out (device double,
// nullable) receives the sketch's estimate of ||g||^2.
size_t heavymix_workspace_bytes(int64_t d, int64_t k);
cudaError_t launch_query_heavymix(const float* merged, const HashCoeffs& h, int r, uint32_t c, int64_t d,
                                  int64_t k, uint64_t fill_seed, int64_t* idx_out, float* est_out, double* l2sq_out,
                                  void* workspace, cudaStream_t s, const cudaEvent_t* marks = nullptr);

// Same pipeline with its scratch in a fixed device array (no allocation); est_out required,
// d <= GS_NOALLOC_MAX_DIM.  The first call on a device looks up the array's address.
cudaError_t launch_query_topk_noalloc(const float* merged, const HashCoeffs& h, int r, uint32_t c,
                                      int64_t d, int64_t k, int64_t* idx_out, float* est_out,
                                      cudaStream_t s, const RowStrides& slow);

inline uint64_t bucket_inverse(uint32_t c) { return c > 1 ? ~0ull / c : 0; }  // floor(2^64 / c) unless c is a power of two
inline bool is_pow2(uint32_t c) { return c && !(c & (c - 1)); }

// ---- launches -----------------------------------------------------------------------
// Every kernel of the library is launched with programmatic stream serialization (sm_90+):
// the next kernel in the stream may be scheduled before this one has finished, and it begins
// with grid_begin(), which waits until the grids it depends on have completed and their
// memory is visible (griddepcontrol.wait), then lets its own successor be scheduled
// (griddepcontrol.launch_dependents).  Launch latency and the ramp of the next grid overlap
// the tail of the previous one; no kernel touches memory before its wait.  A kernel launched
// after a memset, an event record or another library's kernel simply finds its wait satisfied.
__device__ __forceinline__ void grid_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace gs
