// Pieces shared by the resident kernels (resident.cu): the warm start of many
// columns by groups of lanes over entries in global memory, with the values in
// shared memory, and the per-CTA tables they read.
#pragma once

#include <type_traits>

#include "columns.cuh"

namespace imdp {

namespace {

extern __shared__ __align__(16) unsigned char resident_sm[];

// Arrays in the kernel's dynamic shared memory, by offset (a pointer passed
// through a call would lose its address space).
template <class T>
__device__ __forceinline__ T* at_shared(uint32_t off) {
  return reinterpret_cast<T*>(resident_sm + off);
}

// Values V_{k-1} in shared memory, indexed by destination state from `base`:
// 64-bit words, or the high words alone (32-bit storage, whose low words are zero).
struct LocalV {
  uint32_t off;
  int32_t base;
  __device__ __forceinline__ uint64_t at(int32_t r) const { return at_shared<const uint64_t>(off)[r - base]; }
  __device__ __forceinline__ uint32_t hi(int32_t r) const { return (uint32_t)(at(r) >> 32); }
};
struct LocalV32 {
  uint32_t off;
  int32_t base;
  __device__ __forceinline__ uint64_t at(int32_t r) const { return (uint64_t)hi(r) << 32; }
  __device__ __forceinline__ uint32_t hi(int32_t r) const { return at_shared<const uint32_t>(off)[r - base]; }
};

// Columns whose entries are in shared memory too (`gmem` 3 of the column
// routines): destinations and pairs from an offset on.
struct XRows {
  uint32_t off;
  __device__ __forceinline__ int32_t operator[](int idx) const { return at_shared<const int32_t>(off)[idx]; }
};
template <>
struct RowsOf<3> {
  typedef XRows type;
};
template <bool f32>
struct Bounds<f32, 3> {
  uint32_t off;
  int down;
  __device__ __forceinline__ ulonglong2 operator[](int idx) const {
    if (f32) {
      const uint2 m = at_shared<const uint2>(off)[idx];
      return make_ulonglong2((uint64_t)m.x << down, (uint64_t)m.y << down);
    }
    return at_shared<const ulonglong2>(off)[idx];
  }
};

// Entry loads under a predicate; a lane that is off gets destination `none` (a
// valid state) and bounds {0, 0}, which add nothing to any sum.
__device__ __forceinline__ int32_t ld_row_or(const int32_t* p, bool ok, int32_t none) {
  int32_t v;
  asm("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\tmov.b32 %0, %3;\n\t@q ld.global.nc.s32 %0, [%1];\n\t}"
      : "=r"(v)
      : "l"(p), "r"((int)ok), "r"(none));
  return v;
}

// A CTA's columns, longest first (32-bit storage: the 32-bit columns, then the
// correction columns), as a table in shared memory.
struct alignas(16) Col {
  uint64_t rem;   // 1 - sum(lower) (rem_of)
  int32_t a, k;   // first entry (of the model's arrays, or of the CTA's copy), entries
  int32_t e;      // entry the warm start tries (-1: none; 0 when rem = 0, where any will do)
  int32_t hrow;   // its destination
  int32_t x;      // 32-bit storage: shift, or the offset in lgx of a correction column
  uint32_t lc;    // local column, and the flags below
  uint64_t acc;   // a failed warm start's dot product, gap sums below and at the tried key
  uint64_t flt;
  uint64_t geq;
};
constexpr uint32_t kMoving = 0x80000000u;  // the column's last value came from the search (hint -2 - e)
constexpr uint32_t kCarry = 0x40000000u;   // its gaps may add up to 2^64 or more (not narrow_of)
constexpr uint32_t kLocalColumn = 0x3fffffffu;
struct Columns {
  Col* col;
  uint64_t* q;     // by local column: the column's value
  uint16_t* list;  // columns whose warm start failed
};
constexpr int kColumnBytes = (int)sizeof(Col) + 8 + 2;

// Sum over the G lanes of a group (every lane gets it).
template <int G>
__device__ __forceinline__ uint64_t group_sum(uint64_t x) {
  if (G == 32) return warp_sum_u64(x);
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
  return x;
}
template <int G>
__device__ __forceinline__ uint64_t group_sum_sat(uint64_t x) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) x = sat_add(x, __shfl_xor_sync(kFull, x, o));
  return x;
}

// acc + floor(v b / 2^64), from four 32x32-bit products.
__device__ __forceinline__ uint64_t mul_hi_add(uint64_t v, uint64_t b, uint64_t acc) {
  const uint32_t vl = (uint32_t)v, vh = (uint32_t)(v >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
  const uint64_t t1 = (uint64_t)vh * bl + __umulhi(vl, bl);
  const uint64_t t2 = (uint64_t)vl * bh + (uint32_t)t1;
  acc += (uint64_t)vh * bh;
  return acc + ((uint64_t)(uint32_t)(t1 >> 32) + (uint32_t)(t2 >> 32));
}

__device__ __forceinline__ int32_t hint_entry(int32_t h) { return h <= -2 ? -2 - h : h; }

template <bool w64>
struct PairOf {
  typedef uint2 type;
};
template <>
struct PairOf<true> {
  typedef ulonglong2 type;
};
__device__ __forceinline__ uint2 ld_pair(const uint2* p) {
  uint2 v;
  asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ ulonglong2 ld_pair(const ulonglong2* p) {
  ulonglong2 v;
  asm volatile("ld.global.nc.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ int32_t ld_row(const int32_t* p) {
  int32_t v;
  asm volatile("ld.global.nc.s32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ uint2 ld_pair_if(const uint2* p, bool ok) { return ld_stream_u32x2_if(p, ok); }
__device__ __forceinline__ ulonglong2 ld_pair_if(const ulonglong2* p, bool ok) { return ld_stream_u64x2_if(p, ok); }

// Where a lane reads its column's entries: global memory, or the CTA's copy in
// shared memory.
template <class Pair, bool shared>
struct Entries {
  const int32_t* rows;
  const Pair* lg;
  __device__ __forceinline__ int32_t row(int i) const { return ld_row(rows + i); }
  __device__ __forceinline__ Pair pair(int i) const { return ld_pair(lg + i); }
  __device__ __forceinline__ int32_t row_if(int i, bool ok, int32_t none) const { return ld_row_or(rows + i, ok, none); }
  __device__ __forceinline__ Pair pair_if(int i, bool ok) const { return ld_pair_if(lg + i, ok); }
  __device__ __forceinline__ void skip_rows(int n) { rows += n; }
  __device__ __forceinline__ void skip_pairs(int n) { lg += n; }
  __device__ __forceinline__ void skip(int n) {
    rows += n;
    lg += n;
  }
};
template <class Pair>
struct Entries<Pair, true> {
  uint32_t rows, lg;
  __device__ __forceinline__ int32_t row(int i) const { return at_shared<const int32_t>(rows)[i]; }
  __device__ __forceinline__ Pair pair(int i) const { return at_shared<const Pair>(lg)[i]; }
  __device__ __forceinline__ int32_t row_if(int i, bool ok, int32_t none) const { return ok ? row(i) : none; }
  __device__ __forceinline__ Pair pair_if(int i, bool ok) const {
    Pair p{};
    if (ok) p = pair(i);
    return p;
  }
  __device__ __forceinline__ void skip_rows(int n) { rows += n * (uint32_t)sizeof(int32_t); }
  __device__ __forceinline__ void skip_pairs(int n) { lg += n * (uint32_t)sizeof(Pair); }
  __device__ __forceinline__ void skip(int n) {
    skip_rows(n);
    skip_pairs(n);
  }
};

// One lane's sums of the warm pass: acc = sum of V times the chosen bound (the
// upper one below the tried key, else the lower one), chosen = sum of those
// bounds, geq = gap sum at the key. The gap sum below the key is `chosen` less
// the column's sum of lower bounds, which is 1 - rem.
struct WarmSums {
  uint64_t acc, chosen, geq;
};
// `carry`: gap sums may pass 2^64; then `chosen` holds the gap sum below the key
// itself, and both gap sums saturate.
template <bool pess, bool carry>
__device__ __forceinline__ void warm_term(WarmSums& s, uint64_t v, ulonglong2 b, uint64_t vk, int) {
  const bool below = pess ? v < vk : v > vk;
  uint64_t x = b.x;
  if (below) x += b.y;
  s.acc = mul_hi_add(v, x, s.acc);
  if (carry) {
    if (below) s.chosen = sat_add(s.chosen, b.y);
    if (v == vk) s.geq = sat_add(s.geq, b.y);
  } else {
    s.chosen += x;
    if (v == vk) s.geq += b.y;
  }
}
template <bool pess, bool carry>
__device__ __forceinline__ void warm_term(WarmSums& s, uint32_t v, uint2 b, uint32_t vk, int sh) {
  const bool below = pess ? v < vk : v > vk;
  uint32_t x = b.x;
  if (below) x += b.y;  // the upper bound's mantissa, < 2^32
  s.acc += ((uint64_t)v * x) >> sh;
  s.chosen += x;
  if (v == vk) s.geq += b.y;
}
template <bool w64, class VA>
__device__ __forceinline__ typename std::conditional<w64, uint64_t, uint32_t>::type value_of(const VA V, int32_t r) {
  if constexpr (w64)
    return V.at(r);
  else
    return V.hi(r);
}

// U consecutive trips: the loads of all of them are in flight before the first
// is used. `all`: every lane is on in every trip; otherwise trips past `left`
// are not computed and a lane is on while it has entries (`k`) left.
template <int U, bool all, bool w64, int G, bool pess, bool carry, class VA, class Pair, bool shared, class Val>
__device__ __forceinline__ void lane_trips(WarmSums& s, Entries<Pair, shared>& e, int32_t k, int left, const VA V,
                                           Val vk, int sh, int32_t none) {
  int32_t r[U];
  Pair b[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    r[u] = all ? e.row(u * G) : e.row_if(u * G, u * G < k, none);
    b[u] = all ? e.pair(u * G) : e.pair_if(u * G, u * G < k);
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (!all && u > 0 && u >= left) break;
    warm_term<pess, carry>(s, value_of<w64>(V, r[u]), b[u], vk, sh);
  }
  e.skip(U * G);
}

// Entries gl, gl + G, ... of a column (`e` at the lane's first one; `k` entries
// from there). All lanes have `full` trips; `trips` covers the longest column
// of the warp. `none`: any valid state.
template <bool w64, int G, bool pess, bool carry, class VA, class Pair, bool shared>
__device__ __forceinline__ WarmSums lane_sums(Entries<Pair, shared> e, int32_t k, int full, int trips, const VA V,
                                              uint64_t vk64, int sh, int32_t none) {
  typedef typename std::conditional<w64, uint64_t, uint32_t>::type Val;
  const Val vk = w64 ? (Val)vk64 : (Val)(vk64 >> 32);
  WarmSums s{0, 0, 0};
  int t = 0;
  for (; t + 8 <= full; t += 8) lane_trips<8, true, w64, G, pess, carry>(s, e, 0, 0, V, vk, sh, none);
  k -= t * G;
  for (; trips - t > 4; t += 8, k -= 8 * G) lane_trips<8, false, w64, G, pess, carry>(s, e, k, trips - t, V, vk, sh, none);
  if (t < trips) lane_trips<4, false, w64, G, pess, carry>(s, e, k, trips - t, V, vk, sh, none);
  return s;
}

// Warm start (Sec. 4's O-maximization with last iteration's threshold entry) of
// the columns [i0, i1) of the CTA's table, G lanes to a column, 32 / G columns
// to a warp at a time. `w64`: 64-bit bound pairs (64-bit storage, or the
// correction columns of 32-bit storage at their offsets in lgx); otherwise
// 32-bit mantissas in 32-bit arithmetic. The sums are those of warm_pass /
// warm_pass32, so a hit gives the same word; a column that fails, or has no
// hint, goes to the list with its sums.
//
// Bound by instruction issue (the entries come from L2, the values from shared
// memory), so the loop has no predicates up to the shortest column of the warp
// and the gap sum below the key costs no instructions of its own.
template <bool w64, int G, bool pess, bool shared, class VA>
__device__ __forceinline__ void warm_columns(const Columns& C, const Entries<typename PairOf<w64>::type, shared> src,
                                             int i0, int i1, const VA V, bool exact, int32_t none, int warp,
                                             int n_warps, int lane, uint32_t* n_miss) {
  constexpr int NG = 32 / G;
  const int gi = lane / G, gl = lane % G;
  for (int base = i0 + warp * NG; base < i1; base += n_warps * NG) {
    // a group past the end reads the last column along
    Col& c = C.col[min(base + gi, i1 - 1)];
    const uint64_t rem = c.rem;
    const int32_t a = c.a, k = c.k, tried = c.e, hrow = c.hrow, x = c.x;
    const uint32_t lc = c.lc;
    WarmSums s{0, 0, 0};
    uint64_t vk = 0;
    bool narrow = true;
    if (__any_sync(kFull, tried >= 0)) {
      const int full = (int)__reduce_min_sync(kFull, (unsigned)k) / G;
      const int trips = ((int)__reduce_max_sync(kFull, (unsigned)k) + G - 1) / G;
      vk = V.at(hrow);
      if (rem == 0) vk = pess ? 0ull : ~0ull;  // a key no value passes: every entry keeps its lower bound
      Entries<typename PairOf<w64>::type, shared> e = src;
      e.skip_rows(a + gl);
      e.skip_pairs((!shared && w64 && exact ? x : a) + gl);
      if (w64) narrow = !__any_sync(kFull, (lc & kCarry) != 0);
      if (narrow)
        s = lane_sums<w64, G, pess, false>(e, k - gl, full, trips, V, vk, x, none);
      else
        s = lane_sums<w64, G, pess, true>(e, k - gl, full, trips, V, vk, x, none);
      s.acc = group_sum<G>(s.acc);
      if (narrow) {
        s.chosen = group_sum<G>(s.chosen);
        s.geq = group_sum<G>(s.geq);
      } else {
        s.chosen = group_sum_sat<G>(s.chosen);
        s.geq = group_sum_sat<G>(s.geq);
      }
    }
    if (gl == 0 && base + gi < i1) {
      // on 32-bit storage in units of the mantissas: rem and 1 - rem are multiples of 2^(32 - x)
      const uint64_t r = w64 ? rem : rem >> (32 - x), lows = w64 ? kOne - rem : (kOne - rem) >> (32 - x);
      const uint64_t flt = narrow ? s.chosen - lows : s.chosen;
      const uint64_t part = rem == 0 ? 0ull : r - flt;
      if (tried >= 0 && (rem == 0 || (flt < r && part <= s.geq))) {
        C.q[lc & kLocalColumn] = s.acc + (w64 ? __umul64hi(vk, part) : mul_shr(vk >> 32, part, x));
        if (lc & kMoving) c.lc = lc & ~kMoving;
      } else {
        c.acc = s.acc;
        c.flt = flt;
        c.geq = s.geq;
        C.list[atomicAdd(n_miss, 1u)] = (uint16_t)(base + gi);
      }
    }
  }
}

// Loads of the passes below (a lane past the end gets destination `none` and a
// zero pair).
__device__ __forceinline__ int32_t settle_row(GRows rows, int i, bool ok, int32_t none) {
  return ld_row_or(rows.p + i, ok, none);
}
__device__ __forceinline__ int32_t settle_row(XRows rows, int i, bool ok, int32_t none) { return ok ? rows[i] : none; }
template <bool f32>
__device__ __forceinline__ ulonglong2 settle_pair(const Bounds<f32, 1>& lg, int i, bool ok) {
  return lg.at_if(i, ok);
}
template <bool f32>
__device__ __forceinline__ ulonglong2 settle_pair(const Bounds<f32, 3>& lg, int i, bool ok) {
  return ok ? lg[i] : make_ulonglong2(0, 0);
}

// What a warp needs to settle a column, and what the warps of a team exchange.
struct SettleScratch {
  WarpScratch ws;
  unsigned long long x[2][4];  // by parity of the exchange: this warp's partial results
  uint32_t pos;                // the team's candidates
};

// Warps that settle one column together: `size` of them (the first one's scratch
// at `scratch`, the others' behind it), this one's rank, and a barrier of their own.
struct Team {
  int size, rank, bar;
  uint32_t scratch;
  __device__ __forceinline__ SettleScratch* of(int r) const {
    return at_shared<SettleScratch>(scratch + (uint32_t)(r * sizeof(SettleScratch)));
  }
  __device__ __forceinline__ void sync() const {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(32 * size) : "memory");
  }
};

// The team size for `n` missed columns of up to `k` entries on `warps` warps. One
// warp takes 60 cycles for an entry (its passes together) and 6,000 besides, most
// of it waiting for one instruction after the other, so columns that are fewer
// than the warps are shared out; a team's exchanges cost about 6,000 more.
__device__ __forceinline__ int team_size(uint32_t n, int32_t k, int warps) {
  int best = 1;
  uint32_t least = (n + warps - 1) / warps * (45u * (uint32_t)k + 4500u);  // (less a quarter: teams have to pay)
  for (int t = 2; t <= 8 && warps % t == 0; t *= 2) {
    const uint32_t cost = (n * t + warps - 1) / warps * (60u * (uint32_t)k / t + 12000u);
    if (cost < least) {
      least = cost;
      best = t;
    }
  }
  return best;
}

// A column whose warm start failed (or that had no hint), by the whole warp: the
// neighbour check, then the threshold search (the sequence of column_q, to the
// bit). The passes of column_neighbor and column_search load one entry a lane,
// wait, and use it (12 round trips to L2 for 376 entries, and 6 to 12 passes);
// here each pass has the loads of four trips in flight. The neighbour's pass
// takes keys only (its key's entries are looked up by a second one) and leaves
// the key range for the search. Not inlined: the search's registers stay out of
// the warm pass. `none`: any state that V holds.
//
// `team`: by the warps of T, trips dealt round. Their partial results meet in
// shared memory; sums are exact or saturate alike in any order, and candidates are
// ordered by entry, so the words are those of one warp. Grid kernel,
// one warp a column and teams where they pay: cartpole_960 2.54 -> 2.18 ms,
// cartpole_3840 12.8 -> 11.5, 1,712 states of 657 entries 2.13 -> 1.66. The resident
// kernel has columns enough for its warps and its column loop slows down beside the
// second copy of this (4096 pendulum parts 65.2 -> 69.2 ms), so it has one warp each.
template <bool f32, int gmem, int U, bool team, class VA>
__device__ __noinline__ uint64_t missed_column(const typename RowsOf<gmem>::type rows, const Bounds<f32, gmem> lg,
                                               int32_t k, uint64_t rem, const VA V, bool pess, bool neighbor,
                                               uint64_t vk, uint64_t wacc, uint64_t flt, uint64_t geq, const Team T,
                                               int32_t none, int lane, int32_t* hint_out) {
  WarpScratch* ws = &T.of(0)->ws;
  const int size = team ? T.size : 1, rank = team ? T.rank : 0;
  const int step = 32 * size;  // entries from one trip of a warp to its next
  int parity = 0;
  if (team && rank == 0 && lane == 0) T.of(0)->pos = 0;
  // the team's partial results of every warp, one warp's on each of the first lanes
  const auto exchange = [&](uint64_t& a, uint64_t& b, uint64_t& c, uint64_t& d) {
    if (lane == 0) {
      unsigned long long* x = T.of(rank)->x[parity];
      x[0] = a;
      x[1] = b;
      x[2] = c;
      x[3] = d;
    }
    T.sync();
    const unsigned long long* x = T.of(min(lane, size - 1))->x[parity];
    a = x[0];
    b = x[1];
    c = x[2];
    d = x[3];
    parity ^= 1;
  };
  const bool peer = lane < size;  // this lane holds a warp's result after an exchange
  const auto key_of = [&](int32_t r) -> uint64_t {
    const uint64_t v = V.at(r);
    return pess ? v : kOne - v;
  };
  const auto value = [&](uint64_t x) { return pess ? x : kOne - x; };
  // calls f(entry, key) for every entry, a lane's in ascending order
  const auto keys = [&](const auto& f) {
    for (int base = 32 * rank + lane; base < k; base += step * U) {
      int32_t r[U];
#pragma unroll
      for (int u = 0; u < U; ++u) r[u] = settle_row(rows, base + step * u, base + step * u < k, none);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (base + step * u < k) f(base + step * u, key_of(r[u]));
    }
  };
  if (f32 && neighbor) {
    flt = shl_sat(flt, lg.down);
    geq = shl_sat(geq, lg.down);
  }
  const bool down = flt >= rem;
  const uint64_t kap = value(vk);
  uint64_t cmin = ~0ull, cmax = 0, near = down ? 0ull : ~0ull;
  bool have = false;
  keys([&](int, uint64_t x) {
    cmin = x < cmin ? x : cmin;
    cmax = x > cmax ? x : cmax;
    if (down ? x < kap : x > kap) {
      near = down ? (x > near ? x : near) : (x < near ? x : near);
      have = true;
    }
  });
  bool some = __any_sync(kFull, have);
  if (team) {
    uint64_t h = some ? 1 : 0;
    if (neighbor) near = down ? warp_max_u64(near) : warp_min_u64(near);
    cmin = warp_min_u64(cmin);
    cmax = warp_max_u64(cmax);
    exchange(cmin, cmax, near, h);
    some = __any_sync(kFull, peer && h != 0);
  }
  if (neighbor && !(down && flt >= kOne) && some) {
    const uint64_t tgt = down ? warp_max_u64(near) : warp_min_u64(near);
    uint64_t gs = 0, ds = 0, dk = 0;
    int first = -1;
    keys([&](int i, uint64_t x) {
      if (x == tgt || (!down && x == kap)) {
        const ulonglong2 b = lg[i];
        const uint64_t v = value(x), d = __umul64hi(v, b.x + b.y) - __umul64hi(v, b.x);
        if (x == tgt) {
          gs = sat_add(gs, b.y);
          ds += d;
          if (first < 0) first = i;
        } else {
          dk += d;
        }
      }
    });
    uint64_t G = warp_sum_sat(gs), D = warp_sum_u64(ds);
    int32_t h = first;
    if (team) {
      // of the key's entries the one that a single warp's lowest lane sees first
      uint64_t c = __reduce_min_sync(kFull, first >= 0 ? ((unsigned)lane << 26) | ((unsigned)first >> 5) : ~0u);
      dk = warp_sum_u64(dk);
      exchange(G, D, dk, c);
      G = warp_sum_sat(peer ? G : 0);
      D = warp_sum_u64(peer ? D : 0);
      if (!peer) dk = 0;
      const unsigned code = __reduce_min_sync(kFull, (unsigned)c);
      h = (int32_t)(((code & 0x3ffffffu) << 5) | (code >> 26));
    } else {
      h = __shfl_sync(kFull, first, __ffs(__ballot_sync(kFull, first >= 0)) - 1);
    }
    const uint64_t vt = value(tgt);
    if (down) {
      const uint64_t fl = flt - G;
      if (fl < rem) {
        *hint_out = h;
        if (team) T.sync();  // the scratch is free
        return wacc - D + __umul64hi(vt, rem - fl);
      }
    } else {
      const uint64_t DK = warp_sum_u64(dk);
      const uint64_t fl = flt + geq;
      if (sat_add(fl, G) >= rem) {
        *hint_out = h;
        if (team) T.sync();
        return wacc + DK + __umul64hi(vt, rem - fl);
      }
    }
  }
  // threshold search (column_search)
  uint64_t lo = 0, hi = kOne, fb = 0;
  bool all_below = false, uniform = false;
  cmin = warp_min_u64(cmin);
  cmax = warp_max_u64(cmax);
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
    if (!team || rank == 0) {
      ws->hl[lane] = 0;
      ws->hl[lane + 32] = 0;
      ws->hh[lane] = 0;
      ws->hh[lane + 32] = 0;
      ws->hc[lane] = 0;
      ws->hc[lane + 32] = 0;
      if (lane == 0) ws->hsat[0] = ws->hsat[1] = 0;
    }
    if (team)
      T.sync();
    else
      __syncwarp();
    for (int base = 32 * rank + lane; base < k; base += step * U) {
      int32_t r[U];
      uint64_t g[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = base + step * u;
        r[u] = settle_row(rows, i, i < k, none);
        g[u] = settle_pair(lg, i, i < k).y;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (base + step * u >= k) break;
        const uint64_t x = key_of(r[u]);
        if (x >= lo && x <= hi) {
          const int b = (int)((x - cmin) >> shift);
          const uint64_t gg = g[u] < rem ? g[u] : rem;
          const unsigned gl = (unsigned)gg;
          const unsigned old = atomicAdd(&ws->hl[b], gl);
          const unsigned up = (unsigned)(gg >> 32) + ((old + gl) < old ? 1u : 0u);
          if (up) {
            const unsigned oh = atomicAdd(&ws->hh[b], up);
            if (oh + up < oh) atomicOr(&ws->hsat[b >> 5], 1u << (b & 31));
          }
          atomicAdd(&ws->hc[b], 1u);
        }
      }
    }
    if (team)
      T.sync();
    else
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
    const bool low = i0 >= rem;
    const int b = __shfl_sync(kFull, low ? 2 * lane : 2 * lane + 1, L);
    fb = __shfl_sync(kFull, low ? sat_add(fb, ex) : i0, L);
    const unsigned cnt = ws->hc[b];
    if (team)
      T.sync();  // every warp has read the histogram
    else
      __syncwarp();
    lo = cmin + ((uint64_t)b << shift);
    const uint64_t top = lo + ((1ull << shift) - 1ull);
    hi = top < cmax ? top : cmax;
    if (cnt <= 32) break;
    uint64_t a = ~0ull, z = 0;
    keys([&](int, uint64_t x) {
      if (x >= lo && x <= hi) {
        a = x < a ? x : a;
        z = x > z ? x : z;
      }
    });
    cmin = warp_min_u64(a);
    cmax = warp_max_u64(z);
    if (team) {
      uint64_t u0 = 0, u1 = 0;
      exchange(cmin, cmax, u0, u1);
      cmin = warp_min_u64(cmin);
      cmax = warp_max_u64(cmax);
    }
  }
  uint64_t acc = 0, gsum = 0;
  unsigned pos = 0;
  int first_cand = -1;
  const unsigned lt = (1u << lane) - 1u;
  for (int base = 32 * rank; base < k; base += step * U) {
    int32_t r[U];
    ulonglong2 b[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int i = base + step * u + lane;
      r[u] = settle_row(rows, i, i < k, none);
      b[u] = settle_pair(lg, i, i < k);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (base + step * u >= k) break;
      const int i = base + step * u + lane;
      const bool valid = i < k;
      const uint64_t x = key_of(r[u]);
      const bool below = all_below || x < lo;
      const bool cand = valid && !all_below && x >= lo && x <= hi;
      acc = mul_hi_add(value(x), below ? b[u].x + b[u].y : b[u].x, acc);  // past the end: a zero pair
      const unsigned m = __ballot_sync(kFull, cand);
      if (m && first_cand < 0) first_cand = base + step * u + __ffs(m) - 1;
      if (!uniform) {
        if (team && m) {
          if (lane == 0) pos = atomicAdd(&T.of(0)->pos, (unsigned)__popc(m));
          pos = __shfl_sync(kFull, pos, 0);
        }
        if (cand) {
          const unsigned at = min(pos + __popc(m & lt), 31u);
          ws->ck[at] = x;
          ws->cg[at] = b[u].y < rem ? b[u].y : rem;
          ws->ci[at] = i;
        }
        pos += __popc(m);
      } else if (cand) {
        gsum = sat_add(gsum, b[u].y < rem ? b[u].y : rem);
      }
    }
  }
  acc = warp_sum_u64(acc);
  if (team) {
    uint64_t f = (unsigned)first_cand, u1 = 0;
    if (uniform) gsum = warp_sum_sat(gsum);
    exchange(acc, gsum, f, u1);  // (and every warp's candidates are listed)
    acc = warp_sum_u64(peer ? acc : 0);
    if (!peer) gsum = 0;
    first_cand = (int)__reduce_min_sync(kFull, (unsigned)f);
    pos = T.of(0)->pos;
  }
  if (all_below) {
    *hint_out = -1;
    if (team) T.sync();
    return acc;
  }
  pos = min(pos, 32u);
  const uint64_t r2 = rem - fb;  // > 0 by construction of the crossing bin
  if (uniform) {
    const uint64_t g = warp_sum_sat(gsum);
    *hint_out = first_cand >= 0 ? -2 - first_cand : -1;
    if (team) T.sync();
    return acc + __umul64hi(value(lo), g < r2 ? g : r2);
  }
  __syncwarp();
  uint64_t extra = 0;
  int thr = -1;
  if (lane < (int)pos) {
    const uint64_t ki = ws->ck[lane], gi = ws->cg[lane];
    uint64_t before = 0;
    for (unsigned j = 0; j < pos; ++j) {
      const uint64_t kj = ws->ck[j];
      if (kj < ki || (kj == ki && (team ? ws->ci[j] < ws->ci[lane] : j < (unsigned)lane))) before = sat_add(before, ws->cg[j]);
    }
    const uint64_t left = r2 > before ? r2 - before : 0;
    extra = __umul64hi(value(ki), gi < left ? gi : left);
    if (left > 0 && left <= gi) thr = ws->ci[lane];
  }
  const unsigned tm = __ballot_sync(kFull, thr >= 0);
  const int32_t found = tm ? __shfl_sync(kFull, thr, __ffs(tm) - 1) : -1;
  *hint_out = found >= 0 ? -2 - found : -1;
  if (team)
    T.sync();
  else
    __syncwarp();
  return acc + warp_sum_u64(extra);
}

// The CTA's copy of its columns' entries in shared memory (offsets): rows and
// pairs of the columns before n32 (64-bit storage: of all columns) at `pairs`,
// pairs of the correction columns at `exact`, all indexed by the column's `a`.
struct EntryCopy {
  uint32_t rows, pairs, exact;
};

constexpr int kUnitTrips = 2;  // trips in flight while the resident kernel settles a column
// Column i of the table after a failed warm start: its value and hint.
template <bool f32, bool shared, class VA>
__device__ __forceinline__ void settle_column(const Problem& P, const Columns& C, const EntryCopy& D, int i, int n32,
                                              const VA V, uint32_t scratch, int lane) {
  const Col c = C.col[i];
  const uint64_t vk = V.at(c.hrow);
  const bool pess = P.pessimistic != 0, neighbor = c.e >= 0 && !(c.lc & kMoving);
  const int32_t none = shared ? 0 : V.base;
  int32_t ho;
  uint64_t q;
  if constexpr (shared) {
    const XRows rows{D.rows + c.a * 4u};
    if (f32 && i < n32)
      q = missed_column<true, 3, kUnitTrips, false>(rows, Bounds<true, 3>{D.pairs + c.a * 8u, 32 - c.x}, c.k, c.rem, V, pess, neighbor, vk,
                                 c.acc, c.flt, c.geq, Team{1, 0, 0, scratch}, none, lane, &ho);
    else
      q = missed_column<false, 3, kUnitTrips, false>(rows, Bounds<false, 3>{(f32 ? D.exact : D.pairs) + c.a * 16u, 0}, c.k, c.rem, V, pess,
                                  neighbor, vk, c.acc, c.flt, c.geq, Team{1, 0, 0, scratch}, none, lane, &ho);
  } else {
    const GRows rows{P.rowval + c.a};
    if (f32 && i < n32)
      q = missed_column<true, 1, kUnitTrips, false>(rows, Bounds<true, 1>{P.lg32 + c.a, 32 - c.x}, c.k, c.rem, V, pess, neighbor, vk, c.acc,
                                 c.flt, c.geq, Team{1, 0, 0, scratch}, none, lane, &ho);
    else
      q = missed_column<false, 1, kUnitTrips, false>(rows, Bounds<false, 1>{f32 ? P.lgx + c.x : P.lg + c.a, 0}, c.k, c.rem, V, pess,
                                  neighbor, vk, c.acc, c.flt, c.geq, Team{1, 0, 0, scratch}, none, lane, &ho);
  }
  if (lane == 0) {
    const uint32_t lc = c.lc & ~kMoving;
    const int32_t e = hint_entry(ho);
    C.q[lc & kLocalColumn] = q;
    C.col[i].lc = ho <= -2 ? lc | kMoving : lc;
    C.col[i].e = e;
    if (e >= 0) C.col[i].hrow = shared ? XRows{D.rows + c.a * 4u}[e] : __ldg(P.rowval + c.a + e);
  }
  __syncwarp();
}

}  // namespace

}  // namespace imdp
