// Resident Bellman kernel: all iterations of a step call in one launch, for
// problems whose values fit shared memory.
//
// A per-iteration launch reads every transition from HBM, fills and drains the
// whole GPU, and gathers V through L1/L2. Problems are independent of one
// another (and so are the parts of one problem that no transition connects), so
// a thread-block cluster that owns a part can run its iterations back to back:
// it keeps both value buffers, the threshold hints and the column words in
// shared memory, writes each new value into every CTA of the cluster
// (distributed shared memory), and one cluster barrier ends the iteration.
// Transitions are read from global memory every iteration; the cluster size is
// chosen so that the parts in progress together fit L2, so HBM is read about
// once per part instead of once per iteration.
//
// Bound by instruction issue and L2 latency (parts of 240 states, 64-bit storage:
// 50 % issue slots busy, 6.6 TB/s from L2, DRAM 3 % with 1,024 of them under ncu); a transition costs
// 32 warp instructions per 32 lanes, a warp's four columns 290 more. Measured
// against the per-iteration kernels, K = 200: those 4096 parts 115 -> 66 ms
// (32-bit storage 117 -> 66), 256 problems of up to 961 states and horizons from
// 100 to 500 126 -> 70 ms, one problem of 241 states 2.6 -> 0.95 ms per query.
//
// Within a CTA an iteration has three phases: the warm start of the CTA's
// columns by groups of lanes (longest columns first, so the columns that share
// a warp have the same length), the failed columns one at a time with whole
// warps (from a list, so that they spread over the warps), and the states' new
// values. Every column goes through the sums and the sequence of column_q, so
// the words are those of the other kernels.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>

#include "resident.cuh"

namespace imdp {

namespace {

constexpr int kBuckets = 256;  // length classes of the column order: 128 of 32-bit columns, 128 of 64-bit ones

struct ResidentShared {
  Problem prob;  // of the part in progress: read from here (a cluster barrier drops what L1 holds of global memory)
  uint32_t hist[kBuckets];
  uint32_t n_miss[2];  // by iteration parity
  uint32_t n_taken[2];
  unsigned long long resmax[2][kMaxCluster];  // by iteration parity: every rank's max |V_k - V_{k-1}|
  unsigned long long part[32];                // a CTA's maxima by warp
  int32_t unit_next[2];
  int32_t n32;
  int32_t n_cols;
  int32_t copied;    // the columns' entries are in shared memory
  EntryCopy copy;
  int32_t is_last;
};

struct ResidentLayout {
  size_t v, cols, states, ws, data, bytes;
};
__host__ __device__ inline ResidentLayout resident_layout(int32_t states, int32_t cols, int32_t own, int cell, int warps) {
  auto up = [](size_t x) { return (x + 15) & ~size_t(15); };
  ResidentLayout l;
  size_t o = up(sizeof(ResidentShared));
  l.v = o;      o = up(o + 2 * (size_t)states * cell);
  l.cols = o;   o = up(o + (size_t)cols * kColumnBytes);
  l.states = o; o = up(o + (size_t)(own + 1) * sizeof(int32_t));
  l.ws = o;     o = up(o + (size_t)warps * sizeof(WarpScratch));
  l.data = o;  // the rest: the columns' entries, where they fit
  l.bytes = o;
  return l;
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Barrier of the cluster's CTAs (the CTA's own when it is alone); shared-memory
// writes before it, remote ones too, are visible after it.
__device__ __forceinline__ void cluster_sync(int size) {
  if (size == 1) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
  }
}
__device__ __forceinline__ uint32_t remote(const void* p, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void st_remote(uint64_t* p, uint64_t v, int rank) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(remote(p, rank)), "l"(v) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t* p, uint32_t v, int rank) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(remote(p, rank)), "r"(v) : "memory");
}

template <bool f32>
struct CellOf {
  typedef uint64_t type;
  typedef LocalV view;
  static __device__ __forceinline__ uint64_t put(uint64_t w) { return w; }
  static __device__ __forceinline__ uint64_t get(uint64_t c) { return c; }
};
template <>
struct CellOf<true> {  // values of 32-bit storage: the low word is zero
  typedef uint32_t type;
  typedef LocalV32 view;
  static __device__ __forceinline__ uint32_t put(uint64_t w) { return (uint32_t)(w >> 32); }
  static __device__ __forceinline__ uint64_t get(uint32_t c) { return (uint64_t)c << 32; }
};

// The column tables of states [sa, sb) in shared memory, ordered by length
// class, longest first; states the property fixes are left out. Returns the
// number of columns.
template <bool f32, int G>
__device__ int build_columns(const Problem& P, const Columns& C, int32_t* scol, int32_t sa, int32_t sb, int32_t s0,
                             int32_t max_col, ResidentShared& S) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const int32_t c0 = P.stateptr[sa];
  const int32_t unit = max((max_col + 126 * G) / (127 * G), 1) * G;  // entries per length class
  for (int i = tid; i < kBuckets; i += nt) S.hist[i] = 0;
  __syncthreads();
  auto bucket = [&](int32_t c, int32_t k) {
    const int b = 127 - min((k + unit - 1) / unit, 127);
    return f32 && P.xoff && P.xoff[c] >= 0 ? 128 + b : b;
  };
  for (int32_t s = sa + tid; s < sb; s += nt) {
    const int32_t jb = P.stateptr[s], je = P.stateptr[s + 1];
    const bool free_state = P.fixed[s] == 0;
    scol[s - sa] = (jb - c0) | (free_state ? 0 : (int32_t)0x80000000);
    if (free_state)
      for (int32_t c = jb; c < je; ++c) atomicAdd(&S.hist[bucket(c, P.colptr[c + 1] - P.colptr[c])], 1u);
  }
  if (tid == 0) scol[sb - sa] = P.stateptr[sb] - c0;
  __syncthreads();
  if (tid < 32) {  // exclusive prefix of the classes
    uint32_t h[kBuckets / 32], sum = 0;
    for (int i = 0; i < kBuckets / 32; ++i) {
      h[i] = S.hist[tid * (kBuckets / 32) + i];
      sum += h[i];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, incl, o);
      if (tid >= o) incl += y;
    }
    uint32_t at = incl - sum;
    for (int i = 0; i < kBuckets / 32; ++i) {
      S.hist[tid * (kBuckets / 32) + i] = at;
      at += h[i];
    }
    const int total = (int)__shfl_sync(kFull, incl, 31);
    const int n32 = (int)__shfl_sync(kFull, incl - sum, 16);  // first 64-bit class
    if (tid == 0) {
      S.n32 = f32 ? n32 : 0;
      S.n_cols = total;
    }
  }
  __syncthreads();
  const int total = S.n_cols;
  for (int32_t s = sa + tid; s < sb; s += nt) {
    if (P.fixed[s] != 0) continue;
    const int32_t jb = P.stateptr[s], je = P.stateptr[s + 1];
    for (int32_t c = jb; c < je; ++c) {
      const int32_t a = P.colptr[c], k = P.colptr[c + 1] - a;
      const int at = (int)atomicAdd(&S.hist[bucket(c, k)], 1u);
      const int32_t h = P.hint ? P.hint[c] : -1, e = hint_entry(h);
      const uint64_t word = P.rem[c], rem = rem_of(word);
      Col& col = C.col[at];
      col.rem = rem;
      col.a = a;
      col.k = k;
      col.e = rem == 0 ? 0 : (e >= 0 && e < k ? e : -1);
      col.hrow = rem != 0 && e >= 0 && e < k ? P.rowval[a + e] : s0;
      col.lc = (uint32_t)(c - c0) | (h <= -2 ? kMoving : 0u) | (rem != 0 && !narrow_of(word) ? kCarry : 0u);
      col.x = 0;
      if (f32) {
        const int32_t x = P.xoff ? P.xoff[c] : -1;
        col.x = x >= 0 ? x : P.shift[c];
      }
    }
  }
  return total;
}

// Copies the entries of the CTA's columns behind one another into shared memory
// (from offset `off` on, at most `room` bytes), destinations counted from the
// part's first state; the columns' `a` and `hrow` then mean the copy. Leaves
// S.copied = 0 and everything as it is when they do not fit.
template <bool f32>
__device__ void copy_entries(const Problem& P, const Columns& C, int n_cols, int32_t s0, uint32_t off, uint32_t room,
                             ResidentShared& S) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_warps = blockDim.x >> 5;
  const int n32 = S.n32;
  __syncthreads();
  if (warp == 0) {
    uint32_t at = 0, e32 = 0;
    for (int base = 0; base < n_cols; base += 32) {
      const int i = base + lane;
      const uint32_t k = i < n_cols ? (uint32_t)C.col[i].k : 0u;
      uint32_t incl = k;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
      }
      if (i < n_cols) C.col[i].geq = at + incl - k;
      at += __shfl_sync(kFull, incl, 31);
      if (f32 && base < n32) {
        const int last = min(n32 - base, 32) - 1;
        e32 = at - __shfl_sync(kFull, incl, 31) + __shfl_sync(kFull, incl, last);
      }
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
  for (int i = warp; i < n_cols; i += n_warps) {
    const int32_t a = C.col[i].a, k = C.col[i].k;
    const uint32_t at = (uint32_t)C.col[i].geq;
    const bool exact = f32 && i >= n32;
    for (int32_t t = lane; t < k; t += 32) {
      at_shared<int32_t>(D.rows)[at + t] = P.rowval[a + t] - s0;
      if (!f32)
        at_shared<ulonglong2>(D.pairs)[at + t] = P.lg[a + t];
      else if (exact)
        at_shared<ulonglong2>(D.exact + 16u * at)[t] = P.lgx[C.col[i].x + t];
      else
        at_shared<uint2>(D.pairs)[at + t] = P.lg32[a + t];
    }
  }
  __syncthreads();
  for (int i = tid; i < n_cols; i += blockDim.x) {
    C.col[i].a = (int32_t)C.col[i].geq;
    C.col[i].hrow -= s0;
  }
}

// What the iterations of one part read and write; the same for all of them.
struct Part {
  int32_t s0, ns;      // its states
  int32_t sa, sb;      // this rank's
  int n_cols, n32;     // columns of the table, 32-bit ones first
  int size, rank;
  uint32_t v;          // both value buffers in shared memory
  uint32_t scratch;    // this warp's
  int32_t single;      // every state has one action
};

// Iterations k0 .. k1 of a part (all of the cluster's CTAs together); returns
// the last one run, fewer than asked when the residual of an infinite horizon
// falls below the threshold.
template <bool f32, int G, int NT, bool pess, bool copied>
__device__ __forceinline__ int32_t iterate(const Problem& P, const Columns& C, const int32_t* scol, const Part& A,
                                           int32_t k0, int32_t k1, ResidentShared& S) {
  typedef typename CellOf<f32>::type Cell;
  typedef typename CellOf<f32>::view View;
  constexpr int NW = NT / 32;
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
  const int32_t none = copied ? 0 : A.s0;  // the copy counts destinations from the part's first state
  const uint32_t half = (uint32_t)(A.ns * sizeof(Cell));
  const bool infinite = P.infinite != 0;
  const bool extra = infinite || P.policy_mode != 0;
  const int32_t mine = tid < A.sb - A.sa ? scol[tid] : -1;  // the thread's first state: its first column
  int32_t k = k0;
  for (;; ++k) {
    const int par = k & 1;
    const View V{A.v + (par ? 0u : half), none};
    Cell* Vout = at_shared<Cell>(A.v + (par ? half : 0u));
    // 1. warm start of every column
    if (f32) {
      warm_columns<false, G, pess, copied>(C, e32, 0, A.n32, V, false, none, warp, NW, lane, &S.n_miss[par]);
      if (A.n32 < A.n_cols)
        warm_columns<true, G, pess, copied>(C, e64, A.n32, A.n_cols, V, true, none, warp, NW, lane, &S.n_miss[par]);
    } else {
      warm_columns<true, G, pess, copied>(C, e64, 0, A.n_cols, V, false, none, warp, NW, lane, &S.n_miss[par]);
    }
    __syncthreads();
    // 2. the columns it did not decide
    const uint32_t n_miss = S.n_miss[par];
    if (n_miss) {
      for (;;) {
        uint32_t t = 0;
        if (lane == 0) t = atomicAdd(&S.n_taken[par], 1u);
        t = __shfl_sync(kFull, t, 0);
        if (t >= n_miss) break;
        settle_column<f32, copied>(P, C, D, C.list[t], A.n32, V, A.scratch, lane);
      }
      __syncthreads();
    }
    if (tid == 0) S.n_miss[par ^ 1] = S.n_taken[par ^ 1] = 0;
    // 3. the states
    unsigned long long dmax = 0;
    int32_t jb = mine;
    for (int32_t i = tid; i < A.sb - A.sa; i += NT) {
      if (i != tid) jb = scol[i];
      if (jb < 0) continue;  // Eq. 2 fixes reach and avoid states (both buffers hold their values)
      const int32_t s = A.sa + i;
      uint64_t bestq;
      int32_t best = 0;
      if (A.single)
        bestq = C.q[jb];
      else
        best_action(P, jb, scol[i + 1] & 0x7fffffff, [&](int32_t c) { return C.q[c]; }, &bestq, &best);
      const uint64_t vnew = free_state_value(P, s, bestq);
      Cell* to = &Vout[s - A.s0];
      if (A.size == 1)
        *to = CellOf<f32>::put(vnew);
      else
        for (int r = 0; r < A.size; ++r) st_remote(to, CellOf<f32>::put(vnew), r);
      if (extra) {
        if (P.policy_mode == 1)
          P.policy[(size_t)(P.horizon - k) * P.n_states + s] = best;
        else if (P.policy_mode == 2)
          P.policy[s] = best;
        if (infinite) {
          const uint64_t vold = V.at(s - A.s0 + none);
          const uint64_t d = vnew > vold ? vnew - vold : vold - vnew;
          dmax = d > dmax ? d : dmax;
        }
      }
    }
    if (infinite) {
      // this rank's maximum to every rank's table
      const uint64_t m = warp_max_u64(dmax);
      if (lane == 0) S.part[warp] = m;
      __syncthreads();
      if (tid == 0) {
        uint64_t all = 0;
        for (int w = 0; w < NW; ++w) all = S.part[w] > all ? S.part[w] : all;
        uint64_t* to = reinterpret_cast<uint64_t*>(&S.resmax[par][A.rank]);
        if (A.size == 1)
          *to = all;
        else
          for (int r = 0; r < A.size; ++r) st_remote(to, all, r);
      }
    }
    cluster_sync(A.size);
    if (infinite) {
      unsigned long long all = 0;
      for (int r = 0; r < A.size; ++r) all = S.resmax[par][r] > all ? S.resmax[par][r] : all;
      if (all < P.eps_fix && !P.external_stop) break;
    }
    if (k == k1) break;
  }
  return k;
}

template <bool f32, int G, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) bellman_cluster_kernel(StepLaunch L, ResidentPlan R, int32_t n_iters) {
  unsigned char* sm = resident_sm;
  typedef typename CellOf<f32>::type Cell;
  ResidentShared& S = *reinterpret_cast<ResidentShared*>(sm);
  constexpr int NW = NT / 32;
  const ResidentLayout lay = resident_layout(R.cap_states, R.cap_cols, R.cap_own, sizeof(Cell), NW);
  Cell* Vs = reinterpret_cast<Cell*>(sm + lay.v);
  Columns C;
  {
    unsigned char* p = sm + lay.cols;
    const size_t n = R.cap_cols;
    C.col = reinterpret_cast<Col*>(p);
    C.q = reinterpret_cast<uint64_t*>(C.col + n);
    C.list = reinterpret_cast<uint16_t*>(C.q + n);
  }
  int32_t* scol = reinterpret_cast<int32_t*>(sm + lay.states);
  const int tid = threadIdx.x, warp = tid >> 5;
  Part A;
  A.v = (uint32_t)lay.v;
  A.scratch = (uint32_t)(lay.ws + warp * sizeof(WarpScratch));
  const int size = R.cluster, rank = size > 1 ? (int)cluster_rank() : 0;
  A.size = size;
  A.rank = rank;
  A.single = R.single;

  // shared memory of another CTA may be written only once that CTA has started
  cluster_sync(size);
  for (int j = 0;; ++j) {
    // the next part, taken by rank 0 for the whole cluster
    if (rank == 0 && tid == 0) {
      const uint32_t u = atomicAdd(&L.ctl->tile_next, 1u);
      if (size == 1) S.unit_next[j & 1] = (int32_t)u;
      else for (int r = 0; r < size; ++r) st_remote(reinterpret_cast<uint32_t*>(&S.unit_next[j & 1]), u, r);
    }
    cluster_sync(size);
    const int32_t u = S.unit_next[j & 1];
    if (u >= R.n_units) break;
    const ResidentUnit un = R.units[u];
    const Problem& P = S.prob;
    if (tid < (int)(sizeof(Problem) / 4))
      reinterpret_cast<uint32_t*>(&S.prob)[tid] = reinterpret_cast<const uint32_t*>(&L.probs[un.p])[tid];
    __syncthreads();
    IterState it = L.its[un.p];
    // every rank reads the iteration state before rank 0 writes it back (a barrier lies between)
    const int32_t s0 = un.s0, ns = un.s1 - un.s0;
    const int32_t sa = R.bounds[(size_t)u * (size + 1) + rank], sb = R.bounds[(size_t)u * (size + 1) + rank + 1];
    int n_cols = 0;
    if (!it.done) {
      for (int b = 0; b < 2; ++b)
        for (int32_t i = tid; i < ns; i += NT) Vs[(size_t)b * ns + i] = CellOf<f32>::put(P.V[b][s0 + i]);
      n_cols = build_columns<f32, G>(P, C, scol, sa, sb, s0, R.max_col, S);
      copy_entries<f32>(P, C, n_cols, s0, (uint32_t)lay.data, R.smem - (uint32_t)lay.data, S);
      if (tid < 2) S.n_miss[tid] = S.n_taken[tid] = 0;
    }
    cluster_sync(size);
    if (it.done) continue;
    A.s0 = s0;
    A.ns = ns;
    A.sa = sa;
    A.sb = sb;
    A.n_cols = n_cols;
    A.n32 = f32 ? S.n32 : 0;
    // iterations it.iter + 1 .. last (an infinite horizon's cap is its horizon)
    const int32_t last = min(P.horizon, it.iter + n_iters);
    const bool ran = last > it.iter;
    if (ran) {
      const int32_t k0 = it.iter + 1;
      int32_t k;
      if (S.copied)
        k = P.pessimistic ? iterate<f32, G, NT, true, true>(P, C, scol, A, k0, last, S)
                          : iterate<f32, G, NT, false, true>(P, C, scol, A, k0, last, S);
      else
        k = P.pessimistic ? iterate<f32, G, NT, true, false>(P, C, scol, A, k0, last, S)
                          : iterate<f32, G, NT, false, false>(P, C, scol, A, k0, last, S);
      it.iter = k;
      if (P.infinite) {
        unsigned long long all = 0;
        for (int r = 0; r < size; ++r) all = S.resmax[k & 1][r] > all ? S.resmax[k & 1][r] : all;
        if (all < P.eps_fix && !P.external_stop) {
          it.done = 1;
        } else if (k >= P.horizon) {
          it.done = 1;
          it.noconv = 1;
        }
      } else if (k >= P.horizon) {
        it.done = 1;
      }
    } else {
      it.done = 1;  // horizon 0: nothing to run
    }
    if (it.done) it.k_final = it.iter;
    // back to the session's state
    if (ran) {
      for (int b = 0; b < 2; ++b)
        for (int32_t i = sa - s0 + tid; i < sb - s0; i += NT) P.V[b][s0 + i] = CellOf<f32>::get(Vs[(size_t)b * ns + i]);
      if (P.hint) {
        const int32_t c0 = P.stateptr[sa];
        for (int i = tid; i < n_cols; i += NT) {
          const Col& c = C.col[i];
          if (c.rem != 0) P.hint[c0 + (c.lc & kLocalColumn)] = c.lc & kMoving ? -2 - c.e : c.e;
        }
      }
    }
    // parts of one problem are finite-horizon and end alike: the last CTA advances that problem's state
    if (!R.parts && rank == 0 && tid == 0) {
      it.resmax = 0;
      L.its[un.p] = it;
    }
  }

  // the last CTA resets the launch counters (and advances a problem run in parts)
  __syncthreads();
  if (tid == 0) {
    __threadfence();
    S.is_last = atomicAdd(&L.ctl->finished, 1u) == gridDim.x - 1u;
    if (S.is_last) {
      __threadfence();
      if (R.parts) {
        const Problem& P = L.probs[0];
        IterState it = L.its[0];
        if (!it.done) {
          const int32_t kq = min(P.horizon, it.iter + n_iters);
          it.iter = kq;
          if (kq >= P.horizon) {
            it.done = 1;
            it.k_final = kq;
          }
          L.its[0] = it;
        }
      }
      L.ctl->finished = 0;
      L.ctl->tile_next = 0;
    }
  }
}

typedef void (*ClusterKernel)(StepLaunch, ResidentPlan, int32_t);


ClusterKernel cluster_kernel(const ResidentPlan& R) {
  const auto pick = [&](auto is32, auto nt) -> ClusterKernel {
    constexpr bool s32 = decltype(is32)::value;
    constexpr int NT = decltype(nt)::value, MB = kResidentThreads / NT;
    return R.group == 8 ? bellman_cluster_kernel<s32, 8, NT, MB> : bellman_cluster_kernel<s32, 32, NT, MB>;
  };
  typedef std::integral_constant<int, kResidentThreads / 2> Half;
  typedef std::integral_constant<int, kResidentThreads> Whole;
  if (R.threads == kResidentThreads) return R.f32 ? pick(std::true_type{}, Whole{}) : pick(std::false_type{}, Whole{});
  return R.f32 ? pick(std::true_type{}, Half{}) : pick(std::false_type{}, Half{});
}

cudaError_t configure(ClusterKernel k) {
  cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void*>(k), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)kResidentSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(reinterpret_cast<const void*>(k), cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

cudaLaunchConfig_t cluster_config(const ResidentPlan& R, cudaLaunchAttribute* attr, cudaStream_t st) {
  cudaLaunchConfig_t c;
  std::memset(&c, 0, sizeof(c));
  c.gridDim = dim3((unsigned)std::max(1, R.clusters) * R.cluster);
  c.blockDim = dim3(R.threads);
  c.dynamicSmemBytes = R.smem;
  c.stream = st;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = R.cluster;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  c.attrs = attr;
  c.numAttrs = R.cluster > 1 ? 1 : 0;
  return c;
}

}  // namespace

size_t resident_bytes(int32_t states, int32_t cols, int32_t own, bool f32, int32_t threads) {
  return resident_layout(states, cols, own, f32 ? 4 : 8, threads / 32).bytes;
}

// Clusters of this plan's shape that fit the GPU together; sets R.clusters.
cudaError_t resident_prepare(ResidentPlan& R) {
  ClusterKernel k = cluster_kernel(R);
  cudaError_t e = configure(k);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr;
  R.clusters = 1;
  cudaLaunchConfig_t c = cluster_config(R, &attr, nullptr);
  int n = 0;
  if (R.cluster > 1) {
    e = cudaOccupancyMaxActiveClusters(&n, k, &c);
  } else {
    int sms = 152;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, R.threads, R.smem);
    n *= sms;
  }
  if (e != cudaSuccess) return e;
  if (n < 1) return cudaErrorInvalidConfiguration;
  R.clusters = std::min(n, R.n_units);
  return cudaSuccess;
}

cudaError_t launch_bellman_resident(const StepLaunch& L, const ResidentPlan& R, int32_t n_iters, cudaStream_t st) {
  if (n_iters <= 0) return cudaSuccess;
  ClusterKernel k = cluster_kernel(R);
  cudaLaunchAttribute attr;
  cudaLaunchConfig_t c = cluster_config(R, &attr, st);
  return cudaLaunchKernelEx(&c, k, L, R, n_iters);
}

}  // namespace imdp
