// Grid kernel: all iterations of a step call of one problem in one launch of the
// whole GPU (a cooperative launch; one CTA per SM), for problems too large for
// one thread-block cluster.
//
// Every CTA owns the same few chunks of consecutive states in every iteration
// (dealt round-robin, so that regions where many thresholds move are spread over
// the CTAs). Their column words, threshold hints and reach/avoid mask stay in
// shared memory, and so does the window of V_{k-1} that the chunks' columns
// name: consecutive states of an abstraction reach overlapping runs of states,
// and a column's last destination alone may lie outside (an absorbing
// out-of-domain state, say). Warps take the CTA's columns from a counter, longest
// first, for the warm start. Columns it does not decide are settled by the CTA's
// warps when they are few; otherwise they are listed in global memory, and CTAs
// that have finished take them from any list (a few regions hold most of them:
// with each CTA settling its own, 178,000 of 612,000 cycles of a late iteration of
// pimdp_2, run here without the limit on transitions, were spent waiting). One
// barrier of the grid ends an iteration, three when misses were listed.
//
// A per-iteration launch of the direct kernel has a chain of dependent loads in
// front of every tile (tile counter, tile, descriptor, column words, hint entry,
// its value) and gathers V through L1 and L2; here nothing but the entries
// themselves is loaded in the loop, and entries that fit stay in shared memory.
// The warm start streams at 0.8 of the copy bandwidth (harrier, 109,000 of the
// 230,000 cycles of a late iteration; the rest are misses, 20,000 to 76,000 cycles
// each), and misses bound the first iterations of every model. Measured, K = 200 or to
// convergence: 20,000 states of 24 scattered transitions 3.6 -> 1.27 ms,
// cartpole_960 4.8 -> 2.1, harrier 44.1 -> 34.5, cartpole_3840 13.7 -> 11.4.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstring>

#include "resident.cuh"

namespace imdp {

namespace {

constexpr int kGridWarps = kGridThreads / 32;
// Misses that a CTA settles by itself, two rounds of its warps; more are listed
// for all CTAs, which costs two more barriers.
constexpr uint32_t kGridFewMisses = 2 * kGridWarps;
constexpr int32_t kGridMostCols = 5000;  // of one CTA
constexpr int kSettleTrips = 4;  // trips in flight while a missed column is settled
constexpr int kGridBuckets = 256;  // length classes of the column order, as in the resident kernel
constexpr long long kGridWaitCycles = 4000000000ll;  // ~2 s at 2 GHz: bound of the grid barrier's wait

struct alignas(16) GridCol {
  uint64_t rem;   // 1 - sum(lower) (rem_of)
  int32_t a, k;   // first entry (of the model's arrays, or of the CTA's copy), entries
  int32_t e;      // entry the warm start tries (-1: none; 0 when rem = 0)
  int32_t hrow;   // its destination
  int32_t x;      // 32-bit storage: shift, or the offset in lgx of a correction column
  uint32_t lc;    // local column, and flags
  int32_t win;    // window
  int32_t last;   // destination of the last entry when it lies outside the window, else -1
  int32_t c;      // column of the model
};

// A state that the property leaves free, and where its columns' values are.
struct GridState {
  int32_t s, jb, je;  // state; local columns [jb, je)
};

struct GridShared {
  Problem prob;
  GridUnit unit;  // the problem in progress and its CTAs
  uint32_t hist[kGridBuckets];
  uint32_t next[2];  // columns taken: 32-bit ones (or all), correction columns
  unsigned long long part[kGridWarps];
  int32_t n32, n_cols, n_own, n_win;
  uint32_t n_free, n_lc;
  int32_t copied;
  int32_t stall;  // test hook: the unit's first CTA never arrives at its barriers
  EntryCopy copy;
  int32_t ok;
  uint32_t states, v;                  // the unit's layout
  uint32_t n_miss, taken, total;  // the CTA's misses, those taken; all that were listed
  int32_t chunk_s0[kGridMaxChunks], chunk_own[kGridMaxChunks + 1];
  GridWindow win[kGridMaxChunks];  // `off`: byte offset of state 0's (virtual) cell
  int32_t win_at[kGridMaxChunks + 1];  // cells before the window
};

// Shared memory: what every unit has at the same place (the CTA's state, the
// warps' scratch, the columns' first word; the columns' values backwards from the
// end) needs no register in the column loop. Between them the states, the
// windows, and the entries where they fit.
__host__ __device__ constexpr size_t grid_align(size_t x) { return (x + 15) & ~size_t(15); }
constexpr uint32_t kGridScratchAt = (uint32_t)grid_align(sizeof(GridShared));
constexpr uint32_t kGridColumnsAt = (uint32_t)grid_align(kGridScratchAt + kGridWarps * sizeof(SettleScratch));
struct GridLayout {
  uint32_t states, v, data, q;  // `q`: bytes at the end
};
__host__ __device__ inline GridLayout grid_layout(int32_t cols, int32_t own, int32_t cells, int cell) {
  GridLayout l;
  l.states = (uint32_t)grid_align(kGridColumnsAt + (size_t)cols * sizeof(GridCol));
  l.v = (uint32_t)grid_align(l.states + (size_t)own * sizeof(GridState));
  l.data = (uint32_t)grid_align(l.v + (size_t)cells * cell);
  l.q = (uint32_t)grid_align((size_t)cols * sizeof(uint64_t));
  return l;
}

// V in one of the CTA's windows: `off` is where state 0's cell would be.
template <bool f32>
struct WindowV {
  int32_t off;
  __device__ __forceinline__ uint64_t at(int32_t r) const {
    return *reinterpret_cast<const uint64_t*>(resident_sm + (int32_t)(off + r * 8));
  }
  __device__ __forceinline__ uint32_t hi(int32_t r) const { return (uint32_t)(at(r) >> 32); }
};
template <>
struct WindowV<true> {
  int32_t off;
  __device__ __forceinline__ uint32_t hi(int32_t r) const {
    return *reinterpret_cast<const uint32_t*>(resident_sm + (int32_t)(off + r * 4));
  }
  __device__ __forceinline__ uint64_t at(int32_t r) const { return (uint64_t)hi(r) << 32; }
};
// The same, with states outside the window read from global memory.
template <bool f32>
struct AnyV {
  WindowV<f32> w;
  int32_t w0, len;
  const uint64_t* g;
  __device__ __forceinline__ uint64_t at(int32_t r) const {
    return (uint32_t)(r - w0) < (uint32_t)len ? w.at(r) : __ldcg(reinterpret_cast<const unsigned long long*>(g) + r);
  }
  __device__ __forceinline__ uint32_t hi(int32_t r) const { return (uint32_t)(at(r) >> 32); }
};

// V from global memory, written by other CTAs before the last barrier (not by
// the non-coherent path).
struct CoherentV {
  const uint64_t* g;
  __device__ __forceinline__ uint64_t at(int32_t r) const {
    uint64_t v;
    asm volatile("ld.global.u64 %0, [%1];" : "=l"(v) : "l"(g + r));
    return v;
  }
  __device__ __forceinline__ uint32_t hi(int32_t r) const { return (uint32_t)(at(r) >> 32); }
};

// Barrier `n` (1, 2, ...) of the unit's CTAs: writes before it are visible
// after it (read values written by other CTAs past L1). False when the wait
// gave up or another CTA did.
// Split in two: arrive (writes of the CTA before it), wait.
__device__ __forceinline__ void grid_arrive(StepControl* ctl) {
  __threadfence();
  atomicAdd(&ctl->arrived, 1u);
}
__device__ __forceinline__ bool grid_arrived(const StepControl* ctl, uint32_t target) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&ctl->arrived) : "memory");
  return v >= target;
}
// One poll of a wait that began at t0: false when it gave up or another CTA did.
__device__ __forceinline__ bool grid_waiting(StepControl* ctl, long long t0) {
  if (*(volatile unsigned*)&ctl->error) return false;
  if (clock64() - t0 <= kGridWaitCycles) return true;
  atomicExch(&ctl->error, 1u);
  return false;
}
__device__ __forceinline__ bool grid_sync(StepControl* ctl, uint32_t n, GridShared& S) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t target = n * (uint32_t)S.unit.ctas;
    grid_arrive(ctl);
    const long long t0 = clock64();
    int ok = 1;
    for (uint32_t i = 0; !grid_arrived(ctl, target); ++i)
      if ((i & 255) == 255 && !grid_waiting(ctl, t0)) {
        ok = 0;
        break;
      }
    S.ok = ok;
    __threadfence();
  }
  __syncthreads();
  return S.ok != 0;
}

struct GridTable {
  uint32_t end;  // of shared memory
  __device__ __forceinline__ GridCol& col(int i) const { return at_shared<GridCol>(kGridColumnsAt)[i]; }
  __device__ __forceinline__ uint64_t& q(int lc) const { return *at_shared<uint64_t>(end - 8u - 8u * (uint32_t)lc); }
};

// This CTA's place among the unit's, and its part of the miss list.
__device__ __forceinline__ int unit_rank(const GridShared& S) { return (int)blockIdx.x - S.unit.first; }
__device__ __forceinline__ GridMiss* unit_misses(const GridShared& S) {
  return S.unit.misses + (size_t)unit_rank(S) * S.unit.most_cols;
}

template <bool f32, int G>
__device__ void build_grid_columns(const Problem& P, const GridTable& T, GridState* st, int n_chunks, int32_t max_col,
                                   GridShared& S) {
  const int tid = threadIdx.x;
  const int32_t unit = max((max_col + 126 * G) / (127 * G), 1) * G;  // entries per length class
  for (int i = tid; i < kGridBuckets; i += kGridThreads) S.hist[i] = 0;
  if (tid == 0) S.n_free = S.n_lc = 0;
  __syncthreads();
  const int all = S.chunk_own[n_chunks];
  auto bucket = [&](int32_t c, int32_t k) {
    const int b = 127 - min((k + unit - 1) / unit, 127);
    return f32 && P.xoff && P.xoff[c] >= 0 ? 128 + b : b;
  };
  auto chunk_of = [&](int t) {
    int j = 0;
    while (j + 1 < n_chunks && t >= S.chunk_own[j + 1]) ++j;
    return j;
  };
  for (int t = tid; t < all; t += kGridThreads) {
    const int j = chunk_of(t);
    const int32_t s = S.chunk_s0[j] + (t - S.chunk_own[j]);
    if (P.fixed[s] != 0) continue;  // Eq. 2 fixes reach and avoid states (both buffers hold their values)
    const int32_t jb = P.stateptr[s], je = P.stateptr[s + 1];
    const int at = (int)atomicAdd(&S.n_free, 1u);
    const int32_t lc = (int32_t)atomicAdd(&S.n_lc, (uint32_t)(je - jb));
    st[at] = GridState{s, lc, lc + (je - jb)};
    for (int32_t c = jb; c < je; ++c) atomicAdd(&S.hist[bucket(c, P.colptr[c + 1] - P.colptr[c])], 1u);
  }
  __syncthreads();
  if (tid < 32) {
    uint32_t h[kGridBuckets / 32], sum = 0;
    for (int i = 0; i < kGridBuckets / 32; ++i) {
      h[i] = S.hist[tid * (kGridBuckets / 32) + i];
      sum += h[i];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, incl, o);
      if (tid >= o) incl += y;
    }
    uint32_t at = incl - sum;
    for (int i = 0; i < kGridBuckets / 32; ++i) {
      S.hist[tid * (kGridBuckets / 32) + i] = at;
      at += h[i];
    }
    const int total = (int)__shfl_sync(kFull, incl, 31);
    const int n32 = (int)__shfl_sync(kFull, incl - sum, 16);
    if (tid == 0) {
      S.n32 = f32 ? n32 : total;
      S.n_cols = total;
    }
  }
  __syncthreads();
  if (tid == 0) S.n_own = (int32_t)S.n_free;
  for (int t = tid; t < (int)S.n_free; t += kGridThreads) {
    const GridState g = st[t];
    const int32_t s = g.s;
    int j = 0;
    while (j + 1 < n_chunks && !(s >= S.chunk_s0[j] && s - S.chunk_s0[j] < S.chunk_own[j + 1] - S.chunk_own[j])) ++j;
    const int32_t c0 = P.stateptr[s] - g.jb;  // local column of c: c - c0
    const int w = S.n_win == 1 ? 0 : j;
    const int32_t w0 = S.win[w].w0, w1 = w0 + S.win[w].len;
    for (int32_t c = P.stateptr[s]; c < P.stateptr[s + 1]; ++c) {
      const int32_t a = P.colptr[c], k = P.colptr[c + 1] - a;
      const int at = (int)atomicAdd(&S.hist[bucket(c, k)], 1u);
      const int32_t h = P.hint[c], e = hint_entry(h);
      const uint64_t word = P.rem[c], rem = rem_of(word);
      const int32_t last = k > 0 ? P.rowval[a + k - 1] : w0;
      GridCol col;
      col.rem = rem;
      col.a = a;
      col.k = k;
      col.e = rem == 0 ? 0 : (e >= 0 && e < k ? e : -1);
      col.hrow = rem != 0 && e >= 0 && e < k ? P.rowval[a + e] : w0;
      col.lc = (uint32_t)(c - c0) | (h <= -2 ? kMoving : 0u) | (rem != 0 && !narrow_of(word) ? kCarry : 0u);
      col.x = 0;
      if (f32) {
        const int32_t x = P.xoff ? P.xoff[c] : -1;
        col.x = x >= 0 ? x : P.shift[c];
      }
      col.win = w;
      col.c = c;
      col.last = last >= w1 ? last : -1;
      T.col(at) = col;
    }
  }
  __syncthreads();
}

// The columns' entries behind one another in shared memory, where they fit.
template <bool f32>
__device__ void copy_grid_entries(const Problem& P, const GridTable& T, uint32_t off, uint32_t room, GridShared& S) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n_cols = S.n_cols, n32 = S.n32;
  // (q is free until the first iteration: it holds where a column's copy starts)
  if (warp == 0) {
    uint32_t at = 0, e32 = 0;
    for (int base = 0; base < n_cols; base += 32) {
      const int i = base + lane;
      const uint32_t k = i < n_cols ? (uint32_t)T.col(i).k : 0u;
      uint32_t incl = k;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
      }
      if (i < n_cols) T.q(i) = at + incl - k;
      const uint32_t sum = __shfl_sync(kFull, incl, 31);
      if (base < n32) e32 = at + __shfl_sync(kFull, incl, min(n32 - base, 32) - 1);
      at += sum;
    }
    if (lane == 0) {
      const size_t e = at;
      const size_t rows = (4 * e + 15) & ~size_t(15), pairs = f32 ? (8 * (size_t)e32 + 15) & ~size_t(15) : 16 * e;
      const size_t exact = f32 ? 16 * (e - e32) : 0;
      S.copied = rows + pairs + exact <= room ? 1 : 0;
      S.copy.rows = off;
      S.copy.pairs = off + (uint32_t)rows;
      S.copy.exact = off + (uint32_t)(rows + pairs) - 16u * e32;
    }
  }
  __syncthreads();
  if (!S.copied) return;
  const EntryCopy D = S.copy;
  for (int i = warp; i < n_cols; i += kGridWarps) {
    const int32_t a = T.col(i).a, k = T.col(i).k, x = T.col(i).x;
    const uint32_t at = (uint32_t)T.q(i);
    for (int32_t t = lane; t < k; t += 32) {
      at_shared<int32_t>(D.rows)[at + t] = P.rowval[a + t];
      if (!f32)
        at_shared<ulonglong2>(D.pairs)[at + t] = P.lg[a + t];
      else if (i >= n32)
        at_shared<ulonglong2>(D.exact + 16u * at)[t] = P.lgx[x + t];
      else
        at_shared<uint2>(D.pairs)[at + t] = P.lg32[a + t];
    }
  }
  __syncthreads();
  for (int i = tid; i < n_cols; i += kGridThreads) T.col(i).a = (int32_t)T.q(i);
  __syncthreads();
}

// The columns [i0, i1) of the table, taken G-lane groups at a time from
// `next`: the warm start; the columns it does not decide go to the CTA's part
// of the miss list.
template <bool f32, bool w64, int G, bool pess, bool copied>
__device__ __forceinline__ void grid_columns(const Problem& P, const GridTable& T,
                                             const Entries<typename PairOf<w64>::type, copied> src, int i0, int i1,
                                             bool exact, const uint64_t* Vg, int lane, uint32_t* next, GridShared& S) {
  typedef typename PairOf<w64>::type Pair;
  constexpr int NG = 32 / G;
  const int gi = lane / G, gl = lane % G;
  for (;;) {
    int base = 0;
    if (lane == 0) base = (int)atomicAdd(next, (uint32_t)NG);
    base = i0 + __shfl_sync(kFull, base, 0);
    if (base >= i1) break;
    const int i = min(base + gi, i1 - 1);  // a group past the end reads the last column along
    GridCol& c = T.col(i);
    const uint64_t rem = c.rem;
    const int32_t a = c.a, k = c.k, tried = c.e, hrow = c.hrow, x = c.x, last = c.last;
    const uint32_t lc = c.lc;
    const GridWindow win = S.win[c.win];
    WarmSums s{0, 0, 0};
    uint64_t vk = 0;
    bool narrow = true;
    if (__any_sync(kFull, tried >= 0)) {
      const int32_t kk = last >= 0 ? k - 1 : k;
      const int full = (int)__reduce_min_sync(kFull, (unsigned)kk) / G;
      const int trips = ((int)__reduce_max_sync(kFull, (unsigned)kk) + G - 1) / G;
      Entries<Pair, copied> e = src;
      e.skip_rows(a + gl);
      e.skip_pairs((!copied && w64 && exact ? x : a) + gl);
      // the last entry, when its destination is outside the window
      const bool tail = last >= 0 && gl == 0;
      uint64_t tv = 0;
      Pair tb{};
      if (tail) {
        tv = __ldcg(reinterpret_cast<const unsigned long long*>(Vg) + last);
        tb = e.pair(k - 1);
      }
      vk = (uint32_t)(hrow - win.w0) < (uint32_t)win.len
               ? WindowV<f32>{win.off}.at(hrow)
               : __ldcg(reinterpret_cast<const unsigned long long*>(Vg) + hrow);
      if (rem == 0) vk = pess ? 0ull : ~0ull;  // a key no value passes: every entry keeps its lower bound
      if (w64) narrow = !__any_sync(kFull, (lc & kCarry) != 0);
      const WindowV<f32> V{win.off};
      typedef typename std::conditional<w64, uint64_t, uint32_t>::type Val;
      const Val vkv = w64 ? (Val)vk : (Val)(vk >> 32), tvv = w64 ? (Val)tv : (Val)(tv >> 32);
      if (narrow) {
        s = lane_sums<w64, G, pess, false>(e, kk - gl, full, trips, V, vk, x, win.w0);
        if (__any_sync(kFull, tail)) warm_term<pess, false>(s, tvv, tb, vkv, x);
      } else {
        s = lane_sums<w64, G, pess, true>(e, kk - gl, full, trips, V, vk, x, win.w0);
        if (__any_sync(kFull, tail)) warm_term<pess, true>(s, tvv, tb, vkv, x);
      }
      s.acc = group_sum<G>(s.acc);
      if (narrow) {
        s.chosen = group_sum<G>(s.chosen);
        s.geq = group_sum<G>(s.geq);
      } else {
        s.chosen = group_sum_sat<G>(s.chosen);
        s.geq = group_sum_sat<G>(s.geq);
      }
    }
    // on 32-bit storage in units of the mantissas: rem and 1 - rem are multiples of 2^(32 - x)
    const uint64_t r = w64 ? rem : rem >> (32 - x), lows = w64 ? kOne - rem : (kOne - rem) >> (32 - x);
    const uint64_t flt = narrow ? s.chosen - lows : s.chosen;
    const uint64_t part = rem == 0 ? 0ull : r - flt;
    const bool mine = gl == 0 && base + gi < i1;
    const bool hit = tried >= 0 && (rem == 0 || (flt < r && part <= s.geq));
    if (mine && hit) {
      T.q(lc & kLocalColumn) = s.acc + (w64 ? __umul64hi(vk, part) : mul_shr(vk >> 32, part, x));
      if (lc & kMoving) c.lc = lc & ~kMoving;
    }
    if (mine && !hit) {
      GridMiss m;
      m.rem = rem;
      m.vk = vk;
      m.acc = s.acc;
      m.flt = flt;
      m.geq = s.geq;
      m.i = i;
      m.c = c.c;
      m.k = k;
      m.neighbor = tried >= 0 && !(lc & kMoving) ? 1 : 0;
      m.hint = 0;
      m.pad = 0;
      unit_misses(S)[atomicAdd(&S.n_miss, 1u)] = m;
    }
  }
}

// A record of another warp or CTA (written before a fence or barrier).
__device__ __forceinline__ GridMiss load_miss(const GridMiss* p) {
  GridMiss m;
  const uint4* from = reinterpret_cast<const uint4*>(p);
  uint4* to = reinterpret_cast<uint4*>(&m);
#pragma unroll
  for (int i = 0; i < (int)(sizeof(GridMiss) / 16); ++i) to[i] = __ldcg(from + i);
  return m;
}

// Settles one missed column; its value and hint go to its record. `own`: the
// CTA's own column (its table, windows and copy), else another CTA's.
template <bool f32, bool copied, bool team>
__device__ __forceinline__ void settle_own(const Problem& P, const GridTable& T, const EntryCopy& D, GridMiss* at,
                                           const uint64_t* Vg, const Team& W, int lane, const GridShared& S) {
  const GridMiss m = load_miss(at);
  const GridCol& c = T.col(m.i);
  const GridWindow w = S.win[c.win];
  const AnyV<f32> V{WindowV<f32>{w.off}, w.w0, w.len, Vg};
  const bool pess = P.pessimistic != 0, nb = m.neighbor != 0;
  const int32_t a = c.a, x = c.x;
  int32_t ho;
  uint64_t q;
  if constexpr (copied) {
    const XRows rows{D.rows + a * 4u};
    if (f32 && m.i < S.n32)
      q = missed_column<true, 3, kSettleTrips, team>(rows, Bounds<true, 3>{D.pairs + a * 8u, 32 - x}, m.k, m.rem, V, pess, nb, m.vk, m.acc,
                                 m.flt, m.geq, W, w.w0, lane, &ho);
    else
      q = missed_column<false, 3, kSettleTrips, team>(rows, Bounds<false, 3>{(f32 ? D.exact : D.pairs) + a * 16u, 0}, m.k, m.rem, V, pess, nb,
                                  m.vk, m.acc, m.flt, m.geq, W, w.w0, lane, &ho);
  } else {
    const GRows rows{P.rowval + a};
    if (f32 && m.i < S.n32)
      q = missed_column<true, 1, kSettleTrips, team>(rows, Bounds<true, 1>{P.lg32 + a, 32 - x}, m.k, m.rem, V, pess, nb, m.vk, m.acc, m.flt,
                                 m.geq, W, w.w0, lane, &ho);
    else
      q = missed_column<false, 1, kSettleTrips, team>(rows, Bounds<false, 1>{f32 ? P.lgx + x : P.lg + a, 0}, m.k, m.rem, V, pess, nb, m.vk,
                                  m.acc, m.flt, m.geq, W, w.w0, lane, &ho);
  }
  if (lane == 0 && (!team || W.rank == 0)) {
    at->acc = q;
    at->hint = ho;
  }
}
template <bool f32>
__device__ __forceinline__ void settle_other(const Problem& P, GridMiss* at, const uint64_t* Vg, uint32_t scratch,
                                             int lane) {
  const GridMiss m = load_miss(at);
  const CoherentV V{Vg};
  const bool pess = P.pessimistic != 0, nb = m.neighbor != 0;
  const int32_t a = __ldg(P.colptr + m.c);
  const GRows rows{P.rowval + a};
  int32_t ho, x = -1;
  uint64_t q;
  if (f32 && P.xoff) x = __ldg(P.xoff + m.c);
  if (f32 && x < 0)
    q = missed_column<true, 1, kSettleTrips, false>(rows, Bounds<true, 1>{P.lg32 + a, 32 - __ldg(P.shift + m.c)}, m.k, m.rem, V, pess, nb,
                               m.vk, m.acc, m.flt, m.geq, Team{1, 0, 0, scratch}, 0, lane, &ho);
  else
    q = missed_column<false, 1, kSettleTrips, false>(rows, Bounds<false, 1>{f32 ? P.lgx + x : P.lg + a, 0}, m.k, m.rem, V, pess, nb, m.vk,
                                m.acc, m.flt, m.geq, Team{1, 0, 0, scratch}, 0, lane, &ho);
  if (lane == 0) {
    at->acc = q;
    at->hint = ho;
  }
}

// The CTA's missed columns when there are few: by its warps, from a counter in
// shared memory.
template <bool f32, bool copied>
__device__ __forceinline__ void settle_few(const Problem& P, const GridTable& T, const EntryCopy& D, GridMiss* mine,
                                           uint32_t n, const uint64_t* Vg, uint32_t scratch, int lane, GridShared& S) {
  for (;;) {
    uint32_t j = 0;
    if (lane == 0) j = atomicAdd(&S.taken, 1u);
    j = __shfl_sync(kFull, j, 0);
    if (j >= n) break;
    settle_own<f32, copied, false>(P, T, D, mine + j, Vg, Team{1, 0, 0, scratch}, lane, S);
  }
}

// The same by teams of `size` warps. Not inlined: its registers stay out of the
// column loop.
template <bool f32, bool copied>
__device__ __noinline__ void settle_teams(const GridTable T, uint32_t n, const uint64_t* Vg, int size) {
  GridShared& S = *at_shared<GridShared>(0);
  const EntryCopy D = S.copy;
  GridMiss* mine = unit_misses(S);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, at = warp / size;
  const Team W{size, warp % size, 1 + at, kGridScratchAt + (uint32_t)(at * size * sizeof(SettleScratch))};
  for (uint32_t j = at; j < n; j += kGridWarps / size)
    settle_own<f32, copied, true>(S.prob, T, D, mine + j, Vg, W, lane, S);
}

// Missed columns of this iteration, of the CTAs that listed them (`own` of this
// one). First the CTA's own ones; once every CTA has listed its misses or settled
// its few (barrier `target`, waited for by one thread of the CTA), those that are
// left anywhere, until a look at all lists finds none. False when the wait gave up.
template <bool f32, bool copied>
__device__ bool settle_misses(const Problem& P, const GridTable& T, const EntryCopy& D, const uint64_t* Vg,
                              uint32_t scratch, int k, uint32_t target, uint32_t own, int lane, int warp,
                              GridShared& S) {
  const GridUnit& U = S.unit;
  StepControl* ctl = U.ctl;
  const int n_cta = U.ctas, me = unit_rank(S);
  uint32_t* listed = U.steal + (size_t)(k & 1) * 2 * n_cta;  // per CTA: misses listed
  uint32_t* taken = listed + n_cta;
  GridMiss* mine = unit_misses(S);
  while (own) {
    uint32_t j = 0;
    if (lane == 0) j = atomicAdd(&taken[me], 1u);
    j = __shfl_sync(kFull, j, 0);
    if (j >= own) break;
    settle_own<f32, copied, false>(P, T, D, mine + j, Vg, Team{1, 0, 0, scratch}, lane, S);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const long long t0 = clock64();
    int ok = 1;
    for (uint32_t i = 0; !grid_arrived(ctl, target); ++i)
      if ((i & 255) == 255 && !grid_waiting(ctl, t0)) {
        ok = 0;
        break;
      }
    S.ok = ok;
    S.total = __ldcg(&ctl->misses[k & 3]);
    __threadfence();
  }
  __syncthreads();
  if (!S.ok) return false;
  for (bool found = S.total != 0; found;) {
    found = false;
    for (int base = 0; base < n_cta; base += 32) {
      int v = me + 1 + warp * 6 + base + lane;
      v -= (v / n_cta) * n_cta;
      const bool in = base + lane < n_cta && v != me;
      const uint32_t n = in ? __ldcg(&listed[v]) : 0u;
      unsigned m = __ballot_sync(kFull, n != 0 && __ldcg(&taken[v]) < n);
      while (m) {
        const int src = __ffs(m) - 1;
        m &= m - 1;
        const int victim = __shfl_sync(kFull, v, src);
        const uint32_t many = __shfl_sync(kFull, n, src);
        for (;;) {
          uint32_t j = 0;
          if (lane == 0) j = atomicAdd(&taken[victim], 1u);
          j = __shfl_sync(kFull, j, 0);
          if (j >= many) break;
          found = true;
          settle_other<f32>(P, U.misses + (size_t)victim * U.most_cols + j, Vg, scratch, lane);
        }
      }
    }
  }
  return true;
}

template <bool f32, int G, bool pess, bool copied>
__device__ __forceinline__ int32_t grid_iterate(const Problem& P, const GridTable& T, int32_t k0, int32_t k1, GridShared& S) {
  typedef typename std::conditional<f32, uint32_t, uint64_t>::type Cell;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const EntryCopy D = S.copy;
  Entries<ulonglong2, copied> e64;
  Entries<uint2, copied> e32;
  if constexpr (copied) {
    e32 = Entries<uint2, true>{D.rows, D.pairs};
    e64 = Entries<ulonglong2, true>{D.rows, f32 ? D.exact : D.pairs};
  } else {
    e32 = Entries<uint2, false>{P.rowval, P.lg32};
    e64 = Entries<ulonglong2, false>{P.rowval, f32 ? P.lgx : P.lg};
  }
  const uint32_t scratch = kGridScratchAt + warp * (uint32_t)sizeof(SettleScratch);
  const bool infinite = P.infinite != 0, extra = infinite || P.policy_mode != 0;
  const int n32 = S.n32, n_cols = S.n_cols;
  uint32_t barrier = 0;
  int32_t k = k0;
  for (;; ++k) {
    const uint64_t* Vg = P.V[(k - 1) & 1];
    uint64_t* Vout = P.V[k & 1];
    // the windows of V_{k-1} (other CTAs wrote them: past L1), 256 cells to a warp
    // with all its loads in flight: latency bounds this (20,000 states kept whole:
    // 16,400 cycles with one load in flight per thread, 5,300 so)
    int seg = warp;
    for (int w = 0; w < S.n_win; ++w) {
      const int len = S.win[w].len, n_seg = (len + 255) / 256;
      const unsigned long long* from = reinterpret_cast<const unsigned long long*>(Vg) + S.win[w].w0;
      Cell* to = at_shared<Cell>(S.v) + S.win_at[w];
      for (; seg < n_seg; seg += kGridWarps) {
        const int i = seg * 256 + lane;
        unsigned long long v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = i + 32 * u < len ? __ldcg(from + i + 32 * u) : 0ull;
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (i + 32 * u < len) to[i + 32 * u] = f32 ? (Cell)(v[u] >> 32) : (Cell)v[u];
      }
      seg -= n_seg;
    }
    if (tid < 2) S.next[tid] = 0;
    if (tid == 2) S.n_miss = S.taken = 0;
    __syncthreads();
    if (f32) {
      grid_columns<f32, false, G, pess, copied>(P, T, e32, 0, n32, false, Vg, lane, &S.next[0], S);
      if (n32 < n_cols)
        grid_columns<f32, true, G, pess, copied>(P, T, e64, n32, n_cols, true, Vg, lane, &S.next[1], S);
    } else {
      grid_columns<f32, true, G, pess, copied>(P, T, e64, 0, n_cols, false, Vg, lane, &S.next[0], S);
    }
    __syncthreads();
    const uint32_t n_miss = S.n_miss;
    // the states' new values, policy and residual
    const auto states = [&]() {
      unsigned long long dmax = 0;
      const GridState* st = at_shared<GridState>(S.states);
      const int n_own = S.n_own;
      for (int i = tid; i < n_own; i += kGridThreads) {
        const GridState g = st[i];
        const int32_t s = g.s;
        uint64_t bestq;
        int32_t best = 0;
        if (S.unit.single)
          bestq = T.q(g.jb);
        else
          best_action(P, g.jb, g.je, [&](int32_t c) { return T.q(c); }, &bestq, &best);
        const uint64_t vnew = free_state_value(P, s, bestq);
        Vout[s] = vnew;
        if (extra) {
          if (P.policy_mode == 1)
            P.policy[(size_t)(P.horizon - k) * P.n_states + s] = best;
          else if (P.policy_mode == 2)
            P.policy[s] = best;
          if (infinite) {
            const uint64_t vold = __ldcg(reinterpret_cast<const unsigned long long*>(Vg) + s);
            const uint64_t d = vnew > vold ? vnew - vold : vold - vnew;
            dmax = d > dmax ? d : dmax;
          }
        }
      }
      if (infinite) {
        const uint64_t m = warp_max_u64(dmax);
        if (lane == 0) S.part[warp] = m;
        __syncthreads();
        if (tid == 0) {
          unsigned long long all = 0;
          for (int w = 0; w < kGridWarps; ++w) all = S.part[w] > all ? S.part[w] : all;
          atomicMax(&S.unit.ctl->resid[k & 3], all);
        }
      }
    };
    // the columns' values and hints that the misses' records hold
    const auto collect = [&]() {
      for (uint32_t j = tid; j < n_miss; j += kGridThreads) {
        const GridMiss m = load_miss(unit_misses(S) + j);
        GridCol& c = T.col(m.i);
        const uint32_t lc = c.lc & ~kMoving;
        const int32_t e = hint_entry(m.hint);
        T.q(lc & kLocalColumn) = m.acc;
        c.lc = m.hint <= -2 ? lc | kMoving : lc;
        c.e = e;
        if (e >= 0) c.hrow = copied ? XRows{D.rows + c.a * 4u}[e] : __ldg(P.rowval + c.a + e);
      }
      __syncthreads();
    };
    const uint32_t list = n_miss > kGridFewMisses ? n_miss : 0;
    if (n_miss && !list) {
      const int size = team_size(n_miss, S.unit.max_col, kGridWarps);
      if (size > 1)
        settle_teams<f32, copied>(T, n_miss, Vg, size);
      else
        settle_few<f32, copied>(P, T, D, unit_misses(S), n_miss, Vg, scratch, lane, S);
      __syncthreads();
      collect();
    }
    if (!list) states();
    __syncthreads();
    ++barrier;
    if (tid == 0) {
      // this CTA's misses are listed (its part of the iteration is done if there are none)
      const int n_cta = S.unit.ctas, me = unit_rank(S);
      StepControl* ctl = S.unit.ctl;
      uint32_t* steal = S.unit.steal + (size_t)(k & 1) * 2 * n_cta;
      uint32_t* next = S.unit.steal + (size_t)((k + 1) & 1) * 2 * n_cta;
      next[me] = next[n_cta + me] = 0;  // last read before the previous barrier
      if (me == 0) {
        ctl->resid[(k + 1) & 3] = 0;
        ctl->misses[(k + 1) & 3] = 0;
      }
      if (list) atomicAdd(&ctl->misses[k & 3], list);
      steal[me] = list;
      if (!(S.stall && me == 0)) grid_arrive(ctl);
    }
    if (!settle_misses<f32, copied>(P, T, D, Vg, scratch, k, barrier * (uint32_t)S.unit.ctas, list, lane, warp, S)) return -1;
    if (S.total != 0) {
      // every miss is settled after one more barrier; their CTAs finish, and a last one ends the iteration
      if (!grid_sync(S.unit.ctl, ++barrier, S)) return -1;
      if (list) {
        collect();
        states();
      }
      if (!grid_sync(S.unit.ctl, ++barrier, S)) return -1;
    }
    if (infinite && __ldcg(&S.unit.ctl->resid[k & 3]) < P.eps_fix && !P.external_stop) break;
    if (k == k1) break;
  }
  return k;
}

template <bool f32, int G>
__global__ void __launch_bounds__(kGridThreads, 1) bellman_grid_kernel(StepLaunch L, GridPlan R, int32_t n_iters) {
  GridShared& S = *at_shared<GridShared>(0);
  constexpr int cell = f32 ? 4 : 8;
  const int tid = threadIdx.x;
  const Problem& P = S.prob;
  const int2 todo = R.work[blockIdx.x];
  for (int u = todo.x; u < todo.y; ++u) {
    __syncthreads();  // the unit before is done with shared memory
    if (tid < (int)(sizeof(GridUnit) / 4))
      reinterpret_cast<uint32_t*>(&S.unit)[tid] = reinterpret_cast<const uint32_t*>(R.units + u)[tid];
    __syncthreads();
    const GridUnit& U = S.unit;
    if (n_iters == 0 && U.iters == 0) continue;  // not in this launch
    const GridLayout lay = grid_layout(U.most_cols, U.most_own, U.most_cells, cell);
    const uint32_t end = R.smem & ~15u;
    const GridTable T{end};
    if (tid < (int)(sizeof(Problem) / 4))
      reinterpret_cast<uint32_t*>(&S.prob)[tid] = reinterpret_cast<const uint32_t*>(L.probs + U.p)[tid];
    __syncthreads();
    StepControl* ctl = U.ctl;
    const int n_cta = U.ctas;
    IterState it = L.its[U.p];
    const int32_t last = min(P.horizon, it.iter + (n_iters > 0 ? n_iters : U.iters));
    if (!it.done && last > it.iter) {
      const int me = unit_rank(S);
      const int n_chunks = (U.n_chunks - me + n_cta - 1) / n_cta;
      if (tid == 0) {
        int32_t own = 0, cells = 0;
        for (int j = 0; j < n_chunks; ++j) {
          const int g = me + j * n_cta;
          const int32_t a = U.chunk[g], b = U.chunk[g + 1];
          S.chunk_s0[j] = a;
          S.chunk_own[j] = own;
          own += b - a;
          if (U.one_window && j > 0) continue;
          GridWindow w = U.one_window ? GridWindow{0, P.n_states, 0} : U.win[g];
          w.off = (int32_t)lay.v + (cells - w.w0) * cell;
          S.win[j] = w;
          S.win_at[j] = cells;
          cells += w.len;
        }
        S.chunk_own[n_chunks] = own;
        S.states = lay.states;
        S.v = lay.v;
        S.stall = L.stall;
        S.n_win = U.one_window ? min(1, n_chunks) : n_chunks;
      }
      __syncthreads();
      build_grid_columns<f32, G>(P, T, at_shared<GridState>(lay.states), n_chunks, U.max_col, S);
      copy_grid_entries<f32>(P, T, lay.data, end - lay.q - lay.data, S);
      const int32_t k0 = it.iter + 1;
      int32_t k;
      if (S.copied)
        k = P.pessimistic ? grid_iterate<f32, G, true, true>(P, T, k0, last, S)
                          : grid_iterate<f32, G, false, true>(P, T, k0, last, S);
      else
        k = P.pessimistic ? grid_iterate<f32, G, true, false>(P, T, k0, last, S)
                          : grid_iterate<f32, G, false, false>(P, T, k0, last, S);
      if (k >= 0) {
        it.iter = k;
        const bool settled = P.infinite && __ldcg(&ctl->resid[k & 3]) < P.eps_fix && !P.external_stop;
        if (settled || k >= P.horizon) {
          it.done = 1;
          it.noconv = P.infinite && !settled ? 1 : 0;
        }
        // hints back to the problem's state
        for (int i = tid; i < S.n_cols; i += kGridThreads) {
          const GridCol& c = T.col(i);
          if (c.rem == 0) continue;
          P.hint[c.c] = c.lc & kMoving ? -2 - c.e : c.e;
        }
      }
    } else {
      it.done = 1;  // horizon 0: nothing to run
    }
    if (it.done) it.k_final = it.iter;
    __syncthreads();
    // the unit's last CTA writes the iteration state and resets the unit's counters
    // (every CTA has read them by then)
    if (tid == 0) {
      __threadfence();
      if (atomicAdd(&ctl->finished, 1u) == (uint32_t)n_cta - 1u) {
        __threadfence();
        it.resmax = 0;
        L.its[U.p] = it;
        ctl->finished = 0;
        ctl->arrived = 0;
        for (int i = 0; i < 4; ++i) {
          ctl->resid[i] = 0;
          ctl->misses[i] = 0;
        }
      }
    }
  }
}

typedef void (*GridKernel)(StepLaunch, GridPlan, int32_t);

GridKernel grid_kernel(const GridPlan& R) {
  if (R.f32) return R.group == 8 ? bellman_grid_kernel<true, 8> : bellman_grid_kernel<true, 32>;
  return R.group == 8 ? bellman_grid_kernel<false, 8> : bellman_grid_kernel<false, 32>;
}

}  // namespace

size_t grid_bytes(const GridCut& c, bool f32) {
  const GridLayout l = grid_layout(c.most_cols, c.most_own, c.most_cells, f32 ? 4 : 8);
  return (size_t)l.data + l.q;
}

// Fewer CTAs than this cannot hold the model's free columns and states, however it
// is cut (the windows are left out). `columns`: the free ones.
int32_t grid_least_ctas(const DevModel* m, const uint8_t* fx, int64_t* columns) {
  int64_t cols = 0, own = 0;
  for (int32_t s = 0; s < m->n_states; ++s)
    if (!fx[s]) {
      cols += m->h_stateptr[s + 1] - m->h_stateptr[s];
      own += 1;
    }
  *columns = cols;
  const int64_t bytes = cols * (int64_t)(sizeof(GridCol) + sizeof(uint64_t)) + own * (int64_t)sizeof(GridState);
  const int64_t room = (int64_t)kResidentSmem - (int64_t)kGridColumnsAt;
  return (int32_t)std::max<int64_t>({1, (bytes + room - 1) / room, (cols + kGridMostCols - 1) / kGridMostCols});
}

// Cuts the states of a model (`fx`: those the property fixes) into chunks for
// `ctas` CTAs. False when no CTA's share fits.
bool plan_grid_unit(const DevModel* m, const uint8_t* fx, int32_t ctas, GridCut& out) {
  const bool f32 = m->lg32 != nullptr;
  const int32_t n = m->n_states;
  const int32_t* sp = m->h_stateptr.data();
  const int32_t* cp = m->h_colptr.data();
  if (m->h_span.empty() || m->nnz >= kGridMostEntries) return false;
  auto cost = [&](int32_t s) -> int64_t { return fx[s] ? 1 : cp[sp[s + 1]] - cp[sp[s]] + 24 * (sp[s + 1] - sp[s]); };
  int64_t total = 0;
  for (int32_t s = 0; s < n; ++s) total += cost(s);
  // Chunks per CTA: more of them spread the regions where thresholds move (40,000
  // states of 2 actions, 160 MB: 6.8 ms with 8, 5.4 with 16), but each has its own
  // window to load (20,000 states of 40 entries: 1.6 ms with 8, 1.9 with 16): one
  // for every 24 columns, and at most 96 KB of windows. One CTA alone takes all.
  int per = ctas == 1 ? 1
                      : (int)std::min<int64_t>(kGridMaxChunks, std::max<int64_t>(1, m->n_cols / (24 * (int64_t)ctas)));
  std::vector<int64_t> cells, cols, own, ent;
  int64_t most_cells = 0;
  for (;; per = (per + 1) / 2) {
    const int32_t nc = per * ctas;
    out.chunk.assign(nc + 1, 0);
    out.win.assign(nc, GridWindow{});
    cells.assign(ctas, 0);
    cols.assign(ctas, 0);
    own.assign(ctas, 0);
    ent.assign(ctas, 0);
    int64_t done = 0;
    int32_t s = 0;
    for (int32_t g = 0; g < nc; ++g) {
      // states of about equal work, and their window: all their destinations, or
      // all but the columns' last ones when those alone would stretch it
      const int c = g % ctas;
      int32_t lo = n, hi = -1, inner = -1;
      for (; s < n && (g == nc - 1 || done * nc < total * (g + 1)); ++s) {
        done += cost(s);
        lo = std::min(lo, m->h_span[s].x);
        hi = std::max(hi, m->h_span[s].y);
        inner = std::max(inner, m->h_span[s].z);
        if (fx[s]) continue;
        cols[c] += sp[s + 1] - sp[s];
        own[c] += 1;
        ent[c] += cp[sp[s + 1]] - cp[sp[s]];
      }
      out.chunk[g + 1] = s;
      if (hi < 0) lo = hi = 0;
      inner = std::max(inner, lo);
      const int64_t all = (int64_t)hi - lo + 1, most = (int64_t)inner - lo + 1;
      out.win[g] = GridWindow{lo, (int32_t)(all > 2 * most + 64 ? most : all), 0};
      cells[c] += out.win[g].len;
    }
    most_cells = *std::max_element(cells.begin(), cells.end());
    if (per == 1 || most_cells * (f32 ? 4 : 8) <= 96 * 1024 || most_cells >= n) break;
  }
  out.one_window = most_cells >= n ? 1 : 0;
  most_cells = std::min<int64_t>(most_cells, n);
  const int64_t most_cols = *std::max_element(cols.begin(), cols.end());
  const int64_t most_own = *std::max_element(own.begin(), own.end());
  if (most_cells > 60000 || most_cols > kGridMostCols || most_own > 60000) return false;
  out.most_cells = (int32_t)most_cells;
  out.most_cols = (int32_t)most_cols;
  out.most_own = (int32_t)most_own;
  out.entries = *std::max_element(ent.begin(), ent.end());
  return grid_bytes(out, f32) <= kResidentSmem;
}

std::atomic<int> g_refuse_cooperative{0};

cudaError_t grid_prepare(const GridPlan& R) {
  cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(grid_kernel(R)),
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResidentSmem);
  int n = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, grid_kernel(R), kGridThreads, R.smem);
  return e == cudaSuccess && n * bellman_grid() < R.grid ? cudaErrorCooperativeLaunchTooLarge : e;
}

// `n_iters` 0: each unit's own number of iterations.
cudaError_t launch_bellman_grid(const StepLaunch& L, const GridPlan& R, int32_t n_iters, cudaStream_t st) {
  if (n_iters < 0) return cudaSuccess;
  if (g_refuse_cooperative.load(std::memory_order_relaxed)) return cudaErrorCooperativeLaunchTooLarge;
  cudaError_t e = cudaMemsetAsync(R.steal, 0, sizeof(uint32_t) * 4 * (size_t)R.steal_ctas, st);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t c;
  std::memset(&c, 0, sizeof(c));
  c.gridDim = dim3((unsigned)R.grid);
  c.blockDim = dim3(kGridThreads);
  c.dynamicSmemBytes = R.smem;
  c.stream = st;
  cudaLaunchAttribute attr;  // all CTAs resident together: they wait for one another
  attr.id = cudaLaunchAttributeCooperative;
  attr.val.cooperative = 1;
  c.attrs = &attr;
  c.numAttrs = 1;
  StepLaunch l = L;
  l.stall = g_stall_producer.load(std::memory_order_relaxed);
  return cudaLaunchKernelEx(&c, grid_kernel(R), l, R, n_iters);
}

}  // namespace imdp
