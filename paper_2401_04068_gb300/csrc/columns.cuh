// Device routines shared by the Bellman kernels (bellman.cu, resident.cu): exact
// warp sums, the loads of a column's entries, the O-maximization of one column
// (warm start, neighbour check, threshold search; Sec. 4) and the value of a
// state once its actions' values are known (Eq. 2 / Eq. 3). Every kernel runs a
// column through these routines, or through sums of the same exact integer
// terms, so they all give the same words.
#pragma once

#include <cuda_runtime.h>

#include "imdp_internal.h"

namespace imdp {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBins = 64;

// Per-warp scratch. The histogram is dead by the time the candidate list is
// written (the list is filled in the final pass), so the two share storage.
struct WarpScratch {
  union {
    struct {
      unsigned int hl[kBins];    // gap sum per bin, low 32 bits (wraps)
      unsigned int hh[kBins];    // gap sum per bin, high 32 bits plus the low part's carries
      unsigned int hc[kBins];    // entry count per bin
      unsigned int hsat[2];      // bins whose sum passed 2^64 (saturated)
    };
    struct {
      unsigned long long ck[32]; // compacted candidates: key
      unsigned long long cg[32]; //                       gap
      int ci[32];                //                       entry index
    };
  };
};

// ---------------------------------------------------------------- warp reductions

__device__ __forceinline__ uint64_t warp_min_u64(uint64_t x) {
  const unsigned hi = __reduce_min_sync(kFull, (unsigned)(x >> 32));
  const unsigned lo = __reduce_min_sync(kFull, ((unsigned)(x >> 32) == hi) ? (unsigned)x : 0xffffffffu);
  return ((uint64_t)hi << 32) | lo;
}
__device__ __forceinline__ uint64_t warp_max_u64(uint64_t x) {
  const unsigned hi = __reduce_max_sync(kFull, (unsigned)(x >> 32));
  const unsigned lo = __reduce_max_sync(kFull, ((unsigned)(x >> 32) == hi) ? (unsigned)x : 0u);
  return ((uint64_t)hi << 32) | lo;
}
// Exact 64-bit warp sum from three 22/22/20-bit partial sums (no carries lost).
__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t x) {
  const unsigned a = __reduce_add_sync(kFull, (unsigned)(x & 0x3fffffu));
  const unsigned b = __reduce_add_sync(kFull, (unsigned)((x >> 22) & 0x3fffffu));
  const unsigned c = __reduce_add_sync(kFull, (unsigned)(x >> 44));
  return (uint64_t)a + ((uint64_t)b << 22) + ((uint64_t)c << 44);
}

// ---------------------------------------------------------------- saturating sums
//
// Gap sums decide only whether a prefix reaches rem (<= 2^63), and any sum that
// is below rem is needed exactly. So every gap enters the sums clipped to rem
// (which changes no decision: a gap >= rem reaches rem on its own), and sums
// saturate at 2^64 - 1 instead of wrapping (a column's upper bounds may add up
// to far more than 1).

__device__ __forceinline__ uint64_t sat_add(uint64_t a, uint64_t b) {
  const uint64_t c = a + b;
  return c < a ? ~0ull : c;
}
// Warp sum of per-lane values <= 2^63, saturating at 2^64 - 1.
__device__ __forceinline__ uint64_t warp_sum_sat(uint64_t x) {
  x = x > kOne ? kOne : x;
  const unsigned a = __reduce_add_sync(kFull, (unsigned)(x & 0x3fffffu));
  const unsigned b = __reduce_add_sync(kFull, (unsigned)((x >> 22) & 0x1fffffu));
  const unsigned c = __reduce_add_sync(kFull, (unsigned)(x >> 43));
  const unsigned __int128 t = (unsigned __int128)a + ((unsigned __int128)b << 22) + ((unsigned __int128)c << 43);
  return (t >> 64) ? ~0ull : (uint64_t)t;
}
__device__ __forceinline__ uint64_t warp_excl_scan_sat(uint64_t x, int lane) {
  uint64_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl = sat_add(incl, y);
  }
  // exclusive = inclusive of the previous lane
  const uint64_t ex = __shfl_up_sync(kFull, incl, 1);
  return lane == 0 ? 0ull : ex;
}

// ---------------------------------------------------------------- one column

// Entries [0, k) of one column: destinations `rows`, bound pairs `lg` (shared
// or global memory). Keys are recomputed from V on every pass (V is read
// through L1). `hint` is the entry that held the threshold in the previous
// iteration (-1: none); the entry that holds it now is returned in *hint_out.
// Returns q in Q2.62.
//
// Loads from global memory: a column's destinations and bounds (default L1
// policy: a column whose warm start misses is read again by the search, from
// L1), and the values V_{k-1}, gathered by many columns and kept (L1
// evict-last). All of them are read-only during a launch (V_k goes to the
// other buffer), so the non-coherent path is used. A destination or bound load
// guarded by a bounds test in C++ is volatile asm, so that the compiler never
// executes it speculatively ahead of the test (entries past a column's end may
// lie past the end of the array). The gathers of V always read a valid state,
// and the predicated loads below carry their guard inside the asm: those are
// plain asm, which the compiler may schedule freely. (Volatile asm keeps its
// program order, so a volatile gather would hold every later load behind the
// load its address waits for.)
__device__ __forceinline__ int32_t ld_stream_i32(const int32_t* p) {
  int32_t v;
  asm volatile("ld.global.nc.s32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ ulonglong2 ld_stream_u64x2(const ulonglong2* p) {
  ulonglong2 v;
  asm volatile("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ uint2 ld_stream_u32x2(const uint2* p) {
  uint2 v;
  asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ uint64_t ld_value(const uint64_t* p) {
  uint64_t v;
  asm("ld.global.nc.L1::evict_last.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}
// High 32 bits of a value word (the whole value of a problem on 32-bit
// storage, whose values keep their low 32 bits zero).
__device__ __forceinline__ uint32_t ld_value_hi(const uint64_t* p) {
  uint32_t v;
  asm("ld.global.nc.L1::evict_last.u32 %0, [%1];" : "=r"(v) : "l"(reinterpret_cast<const uint32_t*>(p) + 1));
  return v;
}

// The same loads under a predicate: a lane with `ok` false issues no memory
// request and gets zeros (the slice kernel's lanes past their column's end).
// Results come back in 32-bit registers and are assembled after the asm.
__device__ __forceinline__ int32_t ld_stream_i32_if(const int32_t* p, bool ok) {
  int32_t v;
  asm(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\tmov.b32 %0, 0;\n\t@q ld.global.nc.s32 %0, [%1];\n\t}"
      : "=r"(v)
      : "l"(p), "r"((int)ok));
  return v;
}
__device__ __forceinline__ ulonglong2 ld_stream_u64x2_if(const ulonglong2* p, bool ok) {
  uint32_t a, b, c, d;
  asm(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\t"
      "mov.b32 %3, 0;\n\t@q ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "=r"(a), "=r"(b), "=r"(c), "=r"(d)
      : "l"(p), "r"((int)ok));
  return make_ulonglong2(((uint64_t)b << 32) | a, ((uint64_t)d << 32) | c);
}
__device__ __forceinline__ uint2 ld_stream_u32x2_if(const uint2* p, bool ok) {
  uint32_t a, b;
  asm(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %3, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\t"
      "@q ld.global.nc.v2.u32 {%0, %1}, [%2];\n\t}"
      : "=r"(a), "=r"(b)
      : "l"(p), "r"((int)ok));
  return make_uint2(a, b);
}
__device__ __forceinline__ uint64_t ld_value_if(const uint64_t* p, bool ok) {
  uint32_t a, b;
  asm(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %3, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\t"
      "@q ld.global.nc.L1::evict_last.v2.u32 {%0, %1}, [%2];\n\t}"
      : "=r"(a), "=r"(b)
      : "l"(p), "r"((int)ok));
  return ((uint64_t)b << 32) | a;
}
__device__ __forceinline__ uint32_t ld_value_hi_if(const uint64_t* p, bool ok) {
  uint32_t v;
  asm(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\tmov.b32 %0, 0;\n\t"
      "@q ld.global.nc.L1::evict_last.u32 %0, [%1];\n\t}"
      : "=r"(v)
      : "l"(reinterpret_cast<const uint32_t*>(p) + 1), "r"((int)ok));
  return v;
}

// Where the column routines read a column's destinations and bounds (`gmem`):
// 0 shared memory (a plain pointer), 1 contiguous in global memory (streamed
// loads), 2 one column of a slice of the slice layout, whose entry idx sits
// 32 idx slots after its first (streamed loads).
constexpr int kSliceStride = 32;
struct GRows {
  const int32_t* p;
  __device__ __forceinline__ int32_t operator[](int idx) const { return ld_stream_i32(p + idx); }
};
struct SRows {
  const int32_t* p;
  __device__ __forceinline__ int32_t operator[](int idx) const {
    return ld_stream_i32(p + (size_t)idx * kSliceStride);
  }
};
template <int gmem>
struct RowsOf {
  typedef const int32_t* type;
};
template <>
struct RowsOf<1> {
  typedef GRows type;
};
template <>
struct RowsOf<2> {
  typedef SRows type;
};

// Entry idx's destination when `ok`, else 0 (a valid state); from global
// memory a predicated load, which the compiler may schedule freely.
__device__ __forceinline__ int32_t row_if(const int32_t* rows, int idx, bool ok) { return ok ? rows[idx] : 0; }
__device__ __forceinline__ int32_t row_if(GRows rows, int idx, bool ok) { return ld_stream_i32_if(rows.p + idx, ok); }
__device__ __forceinline__ int32_t row_if(SRows rows, int idx, bool ok) {
  return ld_stream_i32_if(rows.p + (size_t)idx * kSliceStride, ok);
}

// Bounds of one column as {lower, gap} in Q1.63, from 64-bit storage or from
// 32-bit mantissas shifted up by `down` = 32 - shift_j; read as `gmem` says.
// `at_if`: entry idx's pair when `ok`, else {0, 0} (predicated in global memory).
template <bool f32, int gmem = 0>
struct Bounds {
  const void* p;
  int down;
  __device__ __forceinline__ ulonglong2 operator[](int idx) const {
    const size_t at = gmem == 2 ? (size_t)idx * kSliceStride : (size_t)idx;
    if (f32) {
      const uint2 m = gmem ? ld_stream_u32x2(static_cast<const uint2*>(p) + at) : static_cast<const uint2*>(p)[at];
      return make_ulonglong2((uint64_t)m.x << down, (uint64_t)m.y << down);
    }
    return gmem ? ld_stream_u64x2(static_cast<const ulonglong2*>(p) + at) : static_cast<const ulonglong2*>(p)[at];
  }
  __device__ __forceinline__ ulonglong2 at_if(int idx, bool ok) const {
    if (gmem == 0) return ok ? (*this)[idx] : make_ulonglong2(0, 0);
    const size_t at = gmem == 2 ? (size_t)idx * kSliceStride : (size_t)idx;
    if (f32) {
      const uint2 m = ld_stream_u32x2_if(static_cast<const uint2*>(p) + at, ok);
      return make_ulonglong2((uint64_t)m.x << down, (uint64_t)m.y << down);
    }
    return ld_stream_u64x2_if(static_cast<const ulonglong2*>(p) + at, ok);
  }
};

// Where the column routines read V_{k-1}: gathers from global memory (the
// tiled kernels; read-only during a launch, L1 evict-last), or from shared
// memory (the single-CTA kernel, which keeps a small problem's values there
// across its iterations). `hi` is the high word, the whole value of a problem
// on 32-bit storage.
struct GlobalV {
  const uint64_t* p;
  __device__ __forceinline__ uint64_t at(int32_t r) const { return ld_value(p + r); }
  __device__ __forceinline__ uint32_t hi(int32_t r) const { return ld_value_hi(p + r); }
};
struct SharedV {
  const uint64_t* p;
  __device__ __forceinline__ uint64_t at(int32_t r) const { return p[r]; }
  __device__ __forceinline__ uint32_t hi(int32_t r) const { return (uint32_t)(p[r] >> 32); }
};

// One pass of the warm start over a column: acc = sum of V times (upper below
// v_k, lower elsewhere), flt = gap sum of the entries below v_k, geq = gap sum of
// the entries at v_k. The trip count is warp-uniform; padding entries read row 0
// and contribute zero. With `carry` the per-lane gap sums count their wraps and
// saturate; without it the column is narrow (all its gaps add up to < 2^64), so
// no sum can wrap.
// Trips of a warm pass from global memory whose loads are in flight ahead of
// the gather being consumed (three measured no faster on 64-bit storage and
// slower on 32-bit, whose deeper unroll then runs short of registers).
constexpr int kPipe = 2;

template <bool carry, bool f32, int gmem, class VP>
__device__ __forceinline__ void warm_pass(const typename RowsOf<gmem>::type rows, const Bounds<f32, gmem> lg, int32_t k,
                                          const VP V, uint64_t vk, bool pess, int lane,
                                          uint64_t& acc, uint64_t& flt, uint64_t& geq) {
  uint32_t fc = 0, gc = 0;
  const int nb = (k + 31) >> 5;
  // from global memory the loop is software-pipelined kPipe trips deep: the
  // destinations and bounds of the next trips are requested before this
  // trip's gather (from shared memory, where the loads are short, the plain
  // loop is faster)
  constexpr bool pipe = gmem != 0;
  int idx = lane;
  int32_t rq[kPipe];
  ulonglong2 bq[kPipe];
#pragma unroll
  for (int d = 0; d < kPipe; ++d) {
    rq[d] = pipe ? row_if(rows, idx + 32 * d, idx + 32 * d < k) : 0;
    bq[d] = pipe ? lg.at_if(idx + 32 * d, idx + 32 * d < k) : make_ulonglong2(0, 0);
  }
  // the gather of the next trip is issued before this trip's arithmetic
  uint64_t vnext = pipe ? V.at(rq[0]) : 0ull;
#pragma unroll 2
  for (int it = 0; it < nb; ++it) {
    if (!pipe) {
      rq[0] = row_if(rows, idx, idx < k);
      bq[0] = lg.at_if(idx, idx < k);
    }
    const ulonglong2 b = bq[0];
    const uint64_t v = pipe ? vnext : V.at(rq[0]);
    idx += 32;
    if (pipe) {
#pragma unroll
      for (int d = 0; d + 1 < kPipe; ++d) {
        rq[d] = rq[d + 1];
        bq[d] = bq[d + 1];
      }
      const int nx = idx + 32 * (kPipe - 1);
      rq[kPipe - 1] = row_if(rows, nx, nx < k);
      bq[kPipe - 1] = lg.at_if(nx, nx < k);
      vnext = V.at(rq[0]);
    }
    const bool below = pess ? (v < vk) : (v > vk);
    acc += __umul64hi(v, b.x + (below ? b.y : 0ull));
    const uint64_t gb = below ? b.y : 0ull, ge = v == vk ? b.y : 0ull;
    flt += gb;
    geq += ge;
    if (carry) {
      fc += flt < gb ? 1u : 0u;
      gc += geq < ge ? 1u : 0u;
    }
  }
  if (carry) {
    flt = fc ? ~0ull : flt;
    geq = gc ? ~0ull : geq;
  }
}

// The warm pass on 32-bit storage, in 32-bit arithmetic (unrolled four trips
// deep: a trip's loads in flight take half the registers of the 64-bit pass's,
// and the deeper unroll keeps twice as many in flight). Values are the high
// words vh (Q1.31) of value words whose low words are zero; bounds are the
// column's mantissas m (value m 2^-(31+s), s = shift_j). Each product vh * m is
// exact in 64 bits, and (vh * m) >> s equals the 64-bit routines' product
// hi64((vh << 32) * (m << (32 - s))) exactly, so this pass gives the same acc,
// and the same decisions from its gap sums (kept in mantissa units, where no
// sum can wrap), as warm_pass on the widened bounds: one 32x32 multiply, a
// shift and a 64-bit add per entry instead of a 64x64 multiply-high.
template <int gmem, class VP>
__device__ __forceinline__ void warm_pass32(const typename RowsOf<gmem>::type rows, const uint2* __restrict__ m,
                                            int32_t k, const VP V, uint32_t vk, int s, bool pess,
                                            int lane, uint64_t& acc, uint64_t& flt, uint64_t& geq) {
  const int nb = (k + 31) >> 5;
  if (gmem == 0) {
#pragma unroll 4
    for (int it = 0; it < nb; ++it) {
      const int idx = it * 32 + lane;
      const bool ok = idx < k;
      const uint32_t v = V.hi(ok ? rows[idx] : 0);
      uint2 b = make_uint2(0, 0);
      if (ok) b = m[idx];
      const bool below = pess ? (v < vk) : (v > vk);
      const uint32_t g = below ? b.y : 0u;
      acc += ((uint64_t)v * (uint64_t)(b.x + g)) >> s;
      flt += g;
      geq += v == vk ? b.y : 0u;
    }
    return;
  }
  // global memory: software-pipelined as in warm_pass
  int idx = lane;
  int32_t rq[kPipe];
  uint2 bq[kPipe];
#pragma unroll
  for (int d = 0; d < kPipe; ++d) {
    rq[d] = row_if(rows, idx + 32 * d, idx + 32 * d < k);
    bq[d] = ld_stream_u32x2_if(m + idx + 32 * d, idx + 32 * d < k);
  }
  uint32_t vnext = V.hi(rq[0]);
#pragma unroll 4
  for (int it = 0; it < nb; ++it) {
    const uint2 b = bq[0];
    const uint32_t v = vnext;
    idx += 32;
#pragma unroll
    for (int d = 0; d + 1 < kPipe; ++d) {
      rq[d] = rq[d + 1];
      bq[d] = bq[d + 1];
    }
    const int nx = idx + 32 * (kPipe - 1);
    rq[kPipe - 1] = row_if(rows, nx, nx < k);
    bq[kPipe - 1] = ld_stream_u32x2_if(m + nx, nx < k);
    vnext = V.hi(rq[0]);
    const bool below = pess ? (v < vk) : (v > vk);
    const uint32_t g = below ? b.y : 0u;
    acc += ((uint64_t)v * (uint64_t)(b.x + g)) >> s;
    flt += g;
    geq += v == vk ? b.y : 0u;
  }
}

// floor(a * b / 2^s) for a < 2^32, b < 2^64, 0 <= s < 64.
__device__ __forceinline__ uint64_t mul_shr(uint64_t a, uint64_t b, int s) {
  const uint64_t lo = a * b, hi = __umul64hi(a, b);
  return s ? (hi << (64 - s)) | (lo >> s) : lo;
}
// x << d, saturating at 2^64 - 1.
__device__ __forceinline__ uint64_t shl_sat(uint64_t x, int d) { return (x >> (64 - d)) ? ~0ull : x << d; }

// `rem_word` is rem = 1 - sum(lower) in Q1.63 (<= 2^63); when 0 < rem < 2^63 and
// the column's gaps add up to < 2^64 ("narrow"), model creation sets bit 63 as a
// flag on top of rem.
__device__ __forceinline__ uint64_t rem_of(uint64_t rem_word) {
  return ((rem_word >> 63) && (rem_word << 1)) ? (rem_word & (kOne - 1)) : rem_word;
}
__device__ __forceinline__ bool narrow_of(uint64_t rem_word) { return (rem_word >> 63) && (rem_word << 1); }

// Warm start. Decides the column without a search when rem = 0 (every entry keeps
// its lower bound) or when last iteration's threshold entry `hint` still holds
// the threshold: with kappa its key it does exactly when F(< kappa) < rem <=
// F(<= kappa), F being the gap sum; then one pass gives q. Comparisons run on V
// itself: key < kappa is V < V_kappa for a pessimistic adversary, V > V_kappa for
// an optimistic one. Returns true with *q set (Q2.62) when decided.
// What a failed warm start leaves for the neighbour check: the tried key's V,
// the pass's dot product and its gap sums below and at that key.
struct WarmMiss {
  uint64_t vk, acc, flt, geq;
  bool valid;
};

template <bool f32, int gmem, class VP>
__device__ __forceinline__ bool column_warm(const typename RowsOf<gmem>::type rows, const Bounds<f32, gmem> lg, int32_t k, uint64_t rem_word,
                                            const VP V, bool pess, int lane, int32_t hint,
                                            uint64_t* q, WarmMiss* miss) {
  miss->valid = false;
  const uint64_t rem = rem_of(rem_word);
  if (rem == 0) {
    uint64_t acc = 0;
#pragma unroll 4
    for (int idx = lane; idx < k; idx += 32) acc += __umul64hi(V.at(rows[idx]), lg[idx].x);
    *q = warp_sum_u64(acc);
    return true;
  }
  if (hint < 0 || hint >= k) return false;
  if (f32) {
    // 32-bit storage: the pass in 32-bit arithmetic (same words as below)
    const int down = lg.down, sh = 32 - down;
    const uint32_t vk32 = V.hi(rows[hint]);
    uint64_t acc = 0, flt = 0, geq = 0;
    warm_pass32<gmem>(rows, static_cast<const uint2*>(lg.p), k, V, vk32, sh, pess, lane, acc, flt, geq);
    acc = warp_sum_u64(acc);
    flt = warp_sum_u64(flt);
    geq = warp_sum_u64(geq);
    const uint64_t rem_m = rem >> down;  // exact: rem is a multiple of 2^down
    if (flt < rem_m && rem_m - flt <= geq) {
      *q = acc + mul_shr(vk32, rem_m - flt, sh);
      return true;
    }
    *miss = WarmMiss{(uint64_t)vk32 << 32, acc, shl_sat(flt, down), shl_sat(geq, down), true};
    return false;
  }
  const uint64_t vk = V.at(rows[hint]);
  uint64_t acc = 0, flt = 0, geq = 0;
  if (narrow_of(rem_word)) {
    // every gap sum of a narrow column is below 2^64: plain exact sums
    warm_pass<false, f32, gmem>(rows, lg, k, V, vk, pess, lane, acc, flt, geq);
    flt = warp_sum_u64(flt);
    geq = warp_sum_u64(geq);
  } else {
    warm_pass<true, f32, gmem>(rows, lg, k, V, vk, pess, lane, acc, flt, geq);
    flt = warp_sum_sat(flt);
    geq = warp_sum_sat(geq);
  }
  acc = warp_sum_u64(acc);
  if (flt < rem && rem - flt <= geq) {
    *q = acc + __umul64hi(vk, rem - flt);
    return true;
  }
  *miss = WarmMiss{vk, acc, flt, geq, true};
  return false;
}

// Neighbour check after a failed warm start at key kappa. If F(< kappa) >= rem the
// threshold lies below kappa, else above it; in most misses it is the adjacent
// distinct key. One pass finds that key (kappa- = the largest key below kappa, or
// kappa+ = the smallest above), the gap sum G of its entries, and the change of
// the warm pass's dot product when the entries between the two keys switch from
// upper to lower bound (or back): D = sum (hi(V (L + G)) - hi(V L)). Then
//   below: F(< kappa-) = F(< kappa) - G, holds when < rem;
//   above: F(< kappa+) = F(<= kappa), holds when F(<= kappa) + G >= rem;
// and q is the warm formula at the new key, to the bit. Returns false when the
// threshold moved further (or a sum is not exact), leaving the full search.
template <bool f32, int gmem, class VP>
__device__ __forceinline__ bool column_neighbor(const typename RowsOf<gmem>::type rows, const Bounds<f32, gmem> lg, int32_t k, uint64_t rem,
                                                const VP V, bool pess, int lane,
                                                const WarmMiss& w, uint64_t* q, int32_t* hint_out) {
  const bool down = w.flt >= rem;
  if (down && w.flt >= kOne) return false;  // F(< kappa) clipped: not exact
  const uint64_t kap = pess ? w.vk : kOne - w.vk;
  uint64_t best = 0, gs = 0, ds = 0, dk = 0;
  bool have = false;
  int32_t bi = -1;
  const int nb = (k + 31) >> 5;
  for (int it = 0; it < nb; ++it) {
    const int idx = it * 32 + lane;
    if (idx >= k) break;
    const uint64_t v = V.at(rows[idx]);
    const uint64_t key = pess ? v : kOne - v;
    const ulonglong2 b = lg[idx];
    const uint64_t d = __umul64hi(v, b.x + b.y) - __umul64hi(v, b.x);
    const bool side = down ? key < kap : key > kap;
    if (side) {
      const bool better = !have || (down ? key > best : key < best);
      if (better) {
        best = key;
        gs = b.y;
        ds = d;
        bi = idx;
        have = true;
      } else if (key == best) {
        gs = sat_add(gs, b.y);
        ds += d;
      }
    } else if (!down && key == kap) {
      dk += d;
    }
  }
  if (!__any_sync(kFull, have)) return false;
  const uint64_t tgt = down ? warp_max_u64(have ? best : 0ull) : warp_min_u64(have ? best : ~0ull);
  const bool mine = have && best == tgt;
  const uint64_t G = warp_sum_sat(mine ? gs : 0ull);
  const uint64_t D = warp_sum_u64(mine ? ds : 0ull);
  const unsigned mm = __ballot_sync(kFull, mine);
  const int32_t h = __shfl_sync(kFull, bi, __ffs(mm) - 1);
  const uint64_t vt = pess ? tgt : kOne - tgt;
  if (down) {
    const uint64_t fl = w.flt - G;  // G <= F(< kappa) < 2^63
    if (fl >= rem) return false;
    *q = w.acc - D + __umul64hi(vt, rem - fl);
  } else {
    const uint64_t DK = warp_sum_u64(dk);
    const uint64_t fl = w.flt + w.geq;  // < rem, exact
    if (sat_add(fl, G) < rem) return false;
    *q = w.acc + DK + __umul64hi(vt, rem - fl);
  }
  *hint_out = h;
  return true;
}

// Threshold search over a column with rem > 0 (the warm start failed or had no
// hint). Returns q in Q2.62 and the threshold entry in *hint_out.
template <bool f32, int gmem, class VP>
__device__ uint64_t column_search(const typename RowsOf<gmem>::type rows, const Bounds<f32, gmem> lg, int32_t k, uint64_t rem_word,
                                  const VP V, bool pess, WarpScratch* ws, int lane,
                                  int32_t* hint_out) {
  const uint64_t rem = rem_of(rem_word);
  auto key_of = [&](int idx) -> uint64_t {
    const uint64_t v = V.at(rows[idx]);
    return pess ? v : (kOne - v);
  };

  // 2. key range
  uint64_t lmin = ~0ull, lmax = 0;
  const int nb = (k + 31) >> 5;
#pragma unroll 4
  for (int it = 0; it < nb; ++it) {
    const int idx = it * 32 + lane;
    if (idx < k) {
      const uint64_t key = key_of(idx);
      lmin = key < lmin ? key : lmin;
      lmax = key > lmax ? key : lmax;
    }
  }
  // 3. threshold search: after it, keys < lo are below (full gap), keys > hi are
  // above (lower bound), keys in [lo, hi] are candidates sharing rem - fb.
  uint64_t lo = 0, hi = kOne, fb = 0;
  bool all_below = false, uniform = false;
  uint64_t cmin = warp_min_u64(lmin), cmax = warp_max_u64(lmax);
  for (int round = 0; round < 12; ++round) {
    if (cmin > cmax) {  // no entry: nothing absorbs rem
      all_below = true;
      break;
    }
    if (cmin == cmax) {  // the candidates share one key
      lo = hi = cmin;
      uniform = true;
      break;
    }
    const int bits = 64 - __clzll((long long)(cmax - cmin));
    const int shift = bits > 6 ? bits - 6 : 0;
    ws->hl[lane] = 0;
    ws->hl[lane + 32] = 0;
    ws->hh[lane] = 0;
    ws->hh[lane + 32] = 0;
    ws->hc[lane] = 0;
    ws->hc[lane + 32] = 0;
    if (lane == 0) ws->hsat[0] = ws->hsat[1] = 0;
    __syncwarp();
    for (int idx = lane; idx < k; idx += 32) {
      const uint64_t key = key_of(idx);
      if (key >= lo && key <= hi) {
        const int b = (int)((key - cmin) >> shift);
        const uint64_t g = lg[idx].y < rem ? lg[idx].y : rem;
        // exact 64-bit bin sums from native 32-bit atomics: the adder whose
        // low-word addition wraps carries one into the high word; a wrap of the
        // high word marks the bin saturated
        const unsigned gl = (unsigned)g;
        const unsigned old = atomicAdd(&ws->hl[b], gl);
        const unsigned up = (unsigned)(g >> 32) + ((old + gl) < old ? 1u : 0u);
        if (up) {
          const unsigned oh = atomicAdd(&ws->hh[b], up);
          if (oh + up < oh) atomicOr(&ws->hsat[b >> 5], 1u << (b & 31));
        }
        atomicAdd(&ws->hc[b], 1u);
      }
    }
    __syncwarp();
    const unsigned sat = ws->hsat[lane >> 4];
    const uint64_t h0 = ((sat >> ((2 * lane) & 31)) & 1u) ? ~0ull
                                                          : (((uint64_t)ws->hh[2 * lane] << 32) | ws->hl[2 * lane]);
    const uint64_t h1 = ((sat >> ((2 * lane + 1) & 31)) & 1u)
                            ? ~0ull
                            : (((uint64_t)ws->hh[2 * lane + 1] << 32) | ws->hl[2 * lane + 1]);
    const uint64_t ex = warp_excl_scan_sat(sat_add(h0, h1), lane);
    const uint64_t i0 = sat_add(sat_add(fb, ex), h0), i1 = sat_add(i0, h1);
    const unsigned cross = __ballot_sync(kFull, i1 >= rem);
    if (cross == 0) {  // first round only: the gaps cannot absorb rem
      all_below = true;
      break;
    }
    const int L = __ffs(cross) - 1;
    const bool first = i0 >= rem;
    const int b = __shfl_sync(kFull, first ? 2 * lane : 2 * lane + 1, L);
    fb = __shfl_sync(kFull, first ? sat_add(fb, ex) : i0, L);  // < rem by the choice of b
    const unsigned cnt = ws->hc[b];
    __syncwarp();
    lo = cmin + ((uint64_t)b << shift);
    const uint64_t top = lo + ((1ull << shift) - 1ull);
    hi = top < cmax ? top : cmax;
    if (cnt <= 32) break;
    // narrow to the min/max of the crossing bin's entries
    uint64_t a = ~0ull, z = 0;
    for (int idx = lane; idx < k; idx += 32) {
      const uint64_t key = key_of(idx);
      if (key >= lo && key <= hi) {
        a = key < a ? key : a;
        z = key > z ? key : z;
      }
    }
    cmin = warp_min_u64(a);
    cmax = warp_max_u64(z);
  }

  // 4. final pass: lower bounds everywhere, full gaps below the candidates,
  // candidates compacted (or summed when they share one key).
  uint64_t acc = 0, gsum = 0;
  unsigned pos = 0;
  int first_cand = -1;
  const unsigned lt = (1u << lane) - 1u;
  for (int base = 0; base < k; base += 32) {
    const int idx = base + lane;
    const bool valid = idx < k;
    uint64_t key = 0;
    ulonglong2 b = make_ulonglong2(0, 0);
    if (valid) {
      key = key_of(idx);
      b = lg[idx];
    }
    const bool below = all_below || key < lo;
    const bool cand = valid && !all_below && key >= lo && key <= hi;
    if (valid) acc += __umul64hi(pess ? key : (kOne - key), below ? b.x + b.y : b.x);
    const unsigned m = __ballot_sync(kFull, cand);
    if (m && first_cand < 0) first_cand = base + __ffs(m) - 1;
    if (!uniform) {
      if (cand) {
        // < 32: a crossing bin of more than 32 entries was narrowed above
        const unsigned at = min(pos + __popc(m & lt), 31u);
        ws->ck[at] = key;
        ws->cg[at] = b.y < rem ? b.y : rem;
        ws->ci[at] = idx;
      }
      pos += __popc(m);
    } else if (cand) {
      gsum = sat_add(gsum, b.y < rem ? b.y : rem);
    }
  }
  acc = warp_sum_u64(acc);
  if (all_below) {
    *hint_out = -1;
    return acc;
  }
  pos = min(pos, 32u);
  const uint64_t r2 = rem - fb;  // > 0 by construction of the crossing bin
  if (uniform) {
    // one key for all candidates: they take min(r2, their total gap) together
    const uint64_t g = warp_sum_sat(gsum);
    *hint_out = first_cand;
    return acc + __umul64hi(pess ? lo : (kOne - lo), g < r2 ? g : r2);
  }
  __syncwarp();
  // Resolve the <= 32 candidates exactly: candidate i takes its gap clipped to
  // what the candidates ordered before it (by key, then list position) leave;
  // the one that takes the last of r2 is the threshold.
  uint64_t extra = 0;
  int thr = -1;
  if (lane < (int)pos) {
    const uint64_t ki = ws->ck[lane], gi = ws->cg[lane];
    uint64_t before = 0;
    for (unsigned j = 0; j < pos; ++j) {
      const uint64_t kj = ws->ck[j];
      if (kj < ki || (kj == ki && j < (unsigned)lane)) before = sat_add(before, ws->cg[j]);
    }
    const uint64_t left = r2 > before ? r2 - before : 0;
    extra = __umul64hi(pess ? ki : (kOne - ki), gi < left ? gi : left);
    if (left > 0 && left <= gi) thr = ws->ci[lane];
  }
  const unsigned tm = __ballot_sync(kFull, thr >= 0);
  *hint_out = tm ? __shfl_sync(kFull, thr, __ffs(tm) - 1) : -1;
  __syncwarp();
  return acc + warp_sum_u64(extra);
}

// One column, warm start first: q in Q2.62, the threshold entry in *hint_out.
template <bool f32, int gmem, class VP>
__device__ uint64_t column_q(const typename RowsOf<gmem>::type rows, const Bounds<f32, gmem> lg, int32_t k, uint64_t rem_word,
                             const VP V, bool pess, WarpScratch* ws, int lane, int32_t hint,
                             int32_t* hint_out) {
  // A hint of -2 - i names entry i as well and records that the column's last
  // value came from the full search: its threshold is moving fast, so a miss
  // goes to the search without trying the neighbour.
  const bool moving = hint <= -2;
  const int32_t entry = moving ? -2 - hint : hint;
  uint64_t q;
  WarmMiss miss;
  if (column_warm<f32, gmem>(rows, lg, k, rem_word, V, pess, lane, entry, &q, &miss)) {
    *hint_out = entry;
    return q;
  }
  if (miss.valid && !moving &&
      column_neighbor<f32, gmem>(rows, lg, k, rem_of(rem_word), V, pess, lane, miss, &q, hint_out))
    return q;
  int32_t found;
  q = column_search<f32, gmem>(rows, lg, k, rem_word, V, pess, ws, lane, &found);
  *hint_out = found >= 0 ? -2 - found : -1;
  return q;
}

__device__ __forceinline__ bool problem_active(const StepLaunch& L, int p, int32_t* k_iter) {
  const IterState& it = L.its[p];
  const Problem& P = L.probs[p];
  *k_iter = it.iter + 1;
  return !it.done && (P.infinite || *k_iter <= P.horizon);
}

// V, policy and residual of state s once its actions' values are known.
__device__ __forceinline__ void finish_state(const Problem& P, int32_t s, int32_t k_iter, uint64_t vnew, int32_t best,
                                             const uint64_t* __restrict__ Vin, uint64_t* __restrict__ Vout,
                                             unsigned long long& dmax) {
  Vout[s] = vnew;
  if (P.policy_mode == 1)
    P.policy[(size_t)(P.horizon - k_iter) * P.n_states + s] = best;
  else if (P.policy_mode == 2)
    P.policy[s] = best;
  if (P.infinite) {
    const uint64_t vold = Vin[s];
    const uint64_t d = vnew > vold ? vnew - vold : vold - vnew;
    dmax = d > dmax ? d : dmax;
  }
}

// Best action of a state over columns [jb, je): first index attaining the optimum.
template <class QAt>
__device__ __forceinline__ void best_action(const Problem& P, int32_t jb, int32_t je, QAt q_at, uint64_t* bestq,
                                            int32_t* best) {
  uint64_t bq = 0;
  int32_t bb = -1;
  for (int32_t jj = jb; jj < je; ++jj) {
    const uint64_t q = q_at(jj);
    if (bb < 0 || (P.maximize ? q > bq : q < bq)) {
      bq = q;
      bb = jj - jb;
    }
  }
  *bestq = bq;
  *best = bb;
}

// V_k(s) of a free state from the optimum over its actions (Q2.62): the
// reachability value clamped at 1, or the reward update W_k = c_s + gamma T(W_{k-1})
// in signed Q2.62, clamped to [0, 1].
// A problem on 32-bit storage keeps its values at 32 bits (rounded to nearest,
// low word zero), which its warm passes read as Q1.31.
__device__ __forceinline__ uint64_t free_state_value(const Problem& P, int32_t s, uint64_t bestq) {
  uint64_t v;
  if (P.property == kPropReward) {
    const int64_t tt = (int64_t)(__umul64hi(P.gamma_fix, bestq) << 1);
    int64_t w = P.rbias[s] + tt;
    w = w < 0 ? 0 : (w > (int64_t)(kOne >> 1) ? (int64_t)(kOne >> 1) : w);
    v = (uint64_t)w << 1;
  } else {
    v = bestq >= (kOne >> 1) ? kOne : (bestq << 1);  // Q2.62 -> Q1.63, clamp at 1
  }
  if (P.lg32) v = round_value32(v);
  return v;
}

}  // namespace

}  // namespace imdp
