// Continuous-batching server: many value-iteration requests (each a resident
// model plus a specification) share the Bellman launches of one slotted batch.
// A worker thread owns the device state; requests are admitted whenever a slot
// and enough of the server's HBM budget are free, join the running batch between
// chunks of iterations, and retire independently when their own horizon or
// convergence test says so. Because every problem's arithmetic is independent
// and exact-integer, a result is the same whether the request ran alone or in
// the mix.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <condition_variable>
#include <cstring>
#include <deque>
#include <map>
#include <mutex>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

#include "imdp_internal.h"

namespace imdp {

namespace {

using Clock = std::chrono::steady_clock;

// V_0 = 1_G in both value buffers (states the property fixes are in no tile,
// so no launch writes them).
__global__ void srv_init_kernel(int32_t n, const uint8_t* __restrict__ fixed, uint64_t* __restrict__ V0) {
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    V0[i] = V0[n + i] = fixed[i] == 1 ? kOne : 0ull;
}

__global__ void srv_export_kernel(int32_t n, const uint64_t* __restrict__ W, double offset, double scale_v,
                                  double* __restrict__ out) {
  const double scale = scale_v / 9223372036854775808.0;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    out[i] = offset + (double)W[i] * scale;
}

// First-fit allocator over one device arena (offsets, 256-byte granules).
class Arena {
 public:
  explicit Arena(size_t bytes) : size_(bytes & ~size_t(255)) { free_[0] = size_; }
  bool alloc(size_t bytes, size_t* off) {
    bytes = (bytes + 255) & ~size_t(255);
    for (auto it = free_.begin(); it != free_.end(); ++it) {
      if (it->second >= bytes) {
        *off = it->first;
        const size_t rest = it->second - bytes, at = it->first + bytes;
        free_.erase(it);
        if (rest) free_[at] = rest;
        return true;
      }
    }
    return false;
  }
  void release(size_t off, size_t bytes) {
    bytes = (bytes + 255) & ~size_t(255);
    auto it = free_.emplace(off, bytes).first;
    auto nx = std::next(it);
    if (nx != free_.end() && it->first + it->second == nx->first) {
      it->second += nx->second;
      free_.erase(nx);
    }
    if (it != free_.begin()) {
      auto pv = std::prev(it);
      if (pv->first + pv->second == it->first) {
        pv->second += it->second;
        free_.erase(it);
      }
    }
  }
  size_t size() const { return size_; }
  size_t largest() const {
    size_t most = 0;
    for (const auto& f : free_) most = std::max(most, f.second);
    return most;
  }

 private:
  size_t size_;
  std::map<size_t, size_t> free_;
};

// Requests running together by rule share launches of the grid kernel: every
// request gets CTAs in proportion to the work it has left, so that all end at
// about the same time, and small ones are run by one CTA one after the other.
// Per-iteration launches of the direct kernel take what the launch and its last
// wave take, 500 times over, while a few large requests hold most of the work
// (64 requests of 50 to 4000 states, 100 to 500 iterations: 49.3 ms,
// 26.5 with shared launches; 1000 requests/s: p50 34 ms and 11 to 16). Bound by the
// misses of the first iterations and by 4 ms of admission and results on the host.
constexpr int32_t kGuessedIterations = 200;
// Thresholds still move in a request's first iterations and most columns miss: a
// launch planned for 2 ms without this took 5.9 with new requests in it, and the
// CTAs of the others waited (the burst of 64 above: 30.2 ms, 26.5 with it).
constexpr int32_t kEarlyIterations = 30;
constexpr double kEarlyCost = 3.0;
// Transitions (and 40 for a column) an SM takes per second: the grid kernel's
// rate on models of 100 and more transitions a column.
constexpr double kEntriesPerSecond = 2.4e9;
// A launch lasts about this long: requests that arrive wait for it, and a launch
// has tables to build (20 to 40 us) and its end to be noticed (50 us).
constexpr double kQuantumSeconds = 2e-3;

struct Request {
  uint64_t ticket = 0;
  DevModel* model = nullptr;
  imdp_spec spec{};
  std::vector<int32_t> reach, avoid;
  std::vector<double> reward;
  Clock::time_point submitted, finished;
  int slot = -1;
  size_t off = 0, bytes = 0;   // arena block
  double v_offset = 0.0, v_scale = 1.0;
  std::vector<double> result;
  int32_t k = 0;
  imdp_status status = IMDP_EPENDING;
  bool done = false;
  std::vector<uint8_t> fixed;  // per state: 1 reach, 2 avoid
  LaunchConfig cfg;            // the server's when the request was admitted
  bool planned = false;        // the two below are set (on the first per-iteration launch)
  std::vector<Tile> tiles;     // tile plan under that configuration (fixed states left out)
  std::vector<int32_t> wide;   // wide states
  // CTAs the grid kernel needs for it, as far as known (0: not looked at). Kept, so
  // that a mix that does not fit is seen at once the next time (12 requests of 300,000
  // columns: 9 cuts of each took 15 ms, again after every arrival and retirement)
  int32_t least = 0;
  int64_t columns = 0;  // free ones, looked at with it
  // iterations left (an infinite horizon: a guess, it ends by itself), and what
  // one of them costs the grid kernel on one SM
  int32_t left() const {
    const int32_t cap = spec.infinite_time ? (spec.horizon > 0 ? spec.horizon : 1000000) : spec.horizon;
    const int32_t n = std::max(cap - k, 1);
    return spec.infinite_time ? std::min(n, kGuessedIterations) : n;
  }
  // `n` iterations from `k` on, the first ones of a request counted several times
  static double weighted(int32_t k, double n) {
    const double early = std::max(0.0, std::min(n, (double)(kEarlyIterations - k)));
    return n + (kEarlyCost - 1.0) * early;
  }
  double work_left() const { return weighted(k, left()); }
  // how many iterations make a weighted number of them (at least)
  int32_t iterations(double w) const {
    const double early = std::max(0, kEarlyIterations - k);
    const double n = w <= early * kEarlyCost ? w / kEarlyCost : early + (w - early * kEarlyCost);
    return (int32_t)std::min<double>(left(), std::max(1.0, std::ceil(n - 1e-9)));
  }
  double seconds(int ctas) const {
    const double work = (double)model->nnz + 40.0 * model->n_cols;
    return (ctas > 1 ? 6.5e-6 : 4e-6) + work / (ctas * kEntriesPerSecond);
  }
};

size_t working_bytes(const DevModel* m, const imdp_spec* sp) {
  const size_t n = (size_t)m->n_states;
  size_t b = 0;
  auto add = [&](size_t x) { b += (x + 255) & ~size_t(255); };
  add(2 * n * sizeof(uint64_t));               // V ping-pong
  add(padded_u8(n));                           // reach/avoid mask
  add(padded_i32(m->n_cols) * sizeof(int32_t));  // threshold hints (padded for bulk copies)
  add(n * sizeof(double));                     // exported values
  if (sp->property == IMDP_REWARD) {
    add(n * sizeof(int64_t));                  // c_s
    add(n * sizeof(uint64_t));                 // W_0
  }
  return b;
}

}  // namespace

struct Server {
  int device = 0;
  int32_t max_active = 1024;
  int32_t chunk = 8;
  Arena arena;
  unsigned char* base = nullptr;
  cudaStream_t stream = nullptr;
  std::mutex mu;
  std::condition_variable cv;
  std::deque<Request*> queue;
  std::map<uint64_t, Request*> all;
  std::vector<Request*> slots;
  uint64_t next_ticket = 1;
  bool stop = false;
  std::thread worker;
  // device tables
  Problem* d_probs = nullptr;
  IterState* d_its = nullptr;
  StepControl* d_ctl = nullptr;
  int32_t* d_base = nullptr;
  Tile* d_tiles = nullptr;
  size_t tile_cap = 0;
  std::vector<Problem> probs_h;
  imdp_status fatal = IMDP_OK;
  LaunchConfig cfg;  // kernel shape and tile plan limits of the launches (worker reads it under mu)
  // statistics (worker thread; read under mu): device time of the chunks (CUDA
  // events around each chunk's launches), wall time of the loop while requests
  // were running, chunks, and requests in the launches summed over chunks
  double st_device_ms = 0.0, st_wall_ms = 0.0, st_slots = 0.0;
  int64_t st_chunks = 0, st_shared = 0;  // all launches (of chunks), and those of the grid kernel
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;

  explicit Server(size_t budget) : arena(budget) {}
  ~Server() {
    {
      std::lock_guard<std::mutex> lk(mu);
      stop = true;
    }
    cv.notify_all();
    if (worker.joinable()) worker.join();
    cudaSetDevice(device);
    if (stream) cudaStreamDestroy(stream);
    cudaFree(base);
    cudaFree(d_probs);
    cudaFree(d_its);
    cudaFree(d_ctl);
    cudaFree(d_base);
    cudaFree(d_tiles);
    cudaFree(d_wide);
    if (ev0) cudaEventDestroy(ev0);
    if (ev1) cudaEventDestroy(ev1);
    side.destroy();
    for (auto& kv : all) delete kv.second;
  }

  // Worker side ------------------------------------------------------------

  bool admit(Request* r, int slot) {
    // called with mu held; sets up device state on the worker stream
    size_t off;
    if (!arena.alloc(r->bytes, &off)) return false;
    r->off = off;
    r->slot = slot;
    const DevModel* m = r->model;
    const int32_t n = m->n_states;
    unsigned char* p = base + off;
    auto take = [&](size_t x) {
      unsigned char* q = p;
      p += (x + 255) & ~size_t(255);
      return q;
    };
    uint64_t* V = (uint64_t*)take(2 * (size_t)n * sizeof(uint64_t));
    uint8_t* mask = take(padded_u8(n));
    int32_t* hints = (int32_t*)take(padded_i32(m->n_cols) * sizeof(int32_t));
    take((size_t)n * sizeof(double));  // export buffer (address recomputed on retire)
    Problem P;
    std::memset(&P, 0, sizeof(P));
    P.stateptr = m->stateptr;
    P.colptr = m->colptr;
    P.rowval = m->rowval;
    P.lg = m->lg;
    P.rem = m->rem;
    P.lg32 = m->lg32;
    P.shift = m->shift;
    P.xoff = m->xoff;
    P.lgx = m->lgx;
    P.fixed = mask;
    P.V[0] = V;
    P.V[1] = V + n;
    P.hint = hints;
    P.n_states = n;
    const imdp_spec* sp = &r->spec;
    P.pessimistic = sp->pessimistic ? 1 : 0;
    P.maximize = sp->maximize ? 1 : 0;
    P.property = sp->property;
    P.infinite = sp->infinite_time ? 1 : 0;
    P.horizon = sp->infinite_time ? (sp->horizon > 0 ? sp->horizon : 1000000) : sp->horizon;
    std::vector<uint8_t>& f = r->fixed;
    f.assign((size_t)n, 0);
    if (sp->property != IMDP_REWARD) {
      for (int32_t v : r->reach) f[v] = 1;
      for (int32_t v : r->avoid) f[v] = 2;
    }
    r->cfg = cfg;
    cudaError_t e = cudaMemsetAsync(mask, 0, padded_u8(n), stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(mask, f.data(), n, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(hints, 0xff, padded_i32(m->n_cols) * sizeof(int32_t), stream);
    if (sp->property == IMDP_REWARD) {
      int64_t* c = (int64_t*)take((size_t)n * sizeof(int64_t));
      uint64_t* w0 = (uint64_t*)take((size_t)n * sizeof(uint64_t));
      double lo, D;
      reward_map(r->reward.data(), n, sp->discount, P.horizon, P.infinite != 0, &lo, &D);
      r->v_offset = lo;
      r->v_scale = D;
      std::vector<int64_t> ch(n);
      std::vector<uint64_t> wh(n);
      for (int32_t s = 0; s < n; ++s) {
        ch[s] = (int64_t)std::llround((r->reward[s] - lo * (1.0 - sp->discount)) / D * 4611686018427387904.0);
        const double ws = std::min(1.0, std::max(0.0, (r->reward[s] - lo) / D));
        wh[s] = (uint64_t)std::llround(ws * 4611686018427387904.0) << 1;
        if (m->lg32) wh[s] = round_value32(wh[s]);  // values of 32-bit storage keep 32 bits
      }
      if (e == cudaSuccess) e = cudaMemcpyAsync(c, ch.data(), sizeof(int64_t) * n, cudaMemcpyHostToDevice, stream);
      if (e == cudaSuccess) e = cudaMemcpyAsync(V, wh.data(), sizeof(uint64_t) * n, cudaMemcpyHostToDevice, stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(stream);  // host vectors go out of scope
      P.rbias = c;
      P.gamma_fix = sp->discount >= 1.0 ? kOne : (uint64_t)std::llround(sp->discount * 9223372036854775808.0);
      P.eps_fix = P.infinite ? eps_fixed(sp->eps / D) : 0;
      (void)w0;
    } else {
      P.eps_fix = P.infinite ? eps_fixed(sp->eps) : 0;
      if (e == cudaSuccess) {
        srv_init_kernel<<<std::min((n + 255) / 256, 1024), 256, 0, stream>>>(n, mask, V);
        e = cudaGetLastError();
      }
    }
    IterState it;
    std::memset(&it, 0, sizeof(it));
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_its + slot, &it, sizeof(it), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);  // `f` and `it` are stack/heap temporaries
    if (e != cudaSuccess) {
      arena.release(r->off, r->bytes);
      r->slot = -1;
      r->status = cuda_status(e, "server admit");
      r->done = true;
      r->finished = Clock::now();
      return true;  // consumed (failed)
    }
    probs_h[slot] = P;
    slots[slot] = r;
    return true;
  }

  imdp_status upload_tables(int32_t count) {
    std::vector<Tile> tiles;
    std::vector<int2> wide;
    int64_t cols = 0;
    for (int32_t s = 0; s < count; ++s) {
      Request* r = slots[s];
      if (!r) continue;
      if (!r->planned) {
        const LaunchConfig rc = resolve_launch(StepLaunch{}, &r->cfg);
        plan_tiles(r->model, 0, r->tiles, r->wide, rc.tile_entries, rc.wide_col, r->fixed.data());
        r->planned = true;
      }
      const size_t at = tiles.size();
      tiles.insert(tiles.end(), r->tiles.begin(), r->tiles.end());
      for (size_t t = at; t < tiles.size(); ++t) {
        tiles[t].p = s;
        cols += tiles[t].c1 - tiles[t].c0;
      }
      for (int32_t st : r->wide) wide.push_back(make_int2(s, st));
    }
    if (wide.size() > wide_cap) {
      cudaFree(d_wide);
      wide_cap = std::max(wide.size(), wide_cap * 2);
      if (cudaMalloc(&d_wide, sizeof(int2) * wide_cap) != cudaSuccess) {
        cudaGetLastError();
        d_wide = nullptr;
        wide_cap = 0;
        set_error("server: wide-state table allocation failed");
        return IMDP_ENOMEM;
      }
    }
    if (tiles.size() > tile_cap) {
      cudaFree(d_tiles);
      tile_cap = std::max(tiles.size(), tile_cap * 2);
      if (cudaMalloc(&d_tiles, sizeof(Tile) * tile_cap) != cudaSuccess) {
        cudaGetLastError();
        d_tiles = nullptr;
        tile_cap = 0;
        set_error("server: tile table allocation failed");
        return IMDP_ENOMEM;
      }
    }
    cudaError_t e = cudaSuccess;
    if (!tiles.empty())
      e = cudaMemcpyAsync(d_tiles, tiles.data(), sizeof(Tile) * tiles.size(), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess && !wide.empty())
      e = cudaMemcpyAsync(d_wide, wide.data(), sizeof(int2) * wide.size(), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return cuda_status(e, "server tables");
    n_tiles = (int32_t)tiles.size();
    n_wide = (int32_t)wide.size();
    tile_cols = cols;
    return IMDP_OK;
  }

  int32_t n_tiles = 0;
  int64_t tile_cols = 0;
  int32_t n_wide = 0;
  SideStream side;
  int2* d_wide = nullptr;
  size_t wide_cap = 0;

  // The grid kernel's plan for the running requests, in a block of the arena
  // (so it counts against the budget; it is given back before requests are admitted).
  GridPlan gplan{};
  size_t g_off = 0, g_bytes = 0;
  std::vector<GridUnit> g_units;  // by CTA; the units of one CTA behind one another
  std::vector<int2> g_work;       // per CTA: its units
  std::vector<Request*> g_reqs;   // per unit
  uint64_t blocked = 0;           // the ticket that waits for budget although no plan held any
  uint64_t launch = 0;            // launches planned
  GridUnit* d_gunits = nullptr;
  int2* d_gwork = nullptr;
  StepControl* d_gctl = nullptr;

  void drop_grid() {
    if (g_bytes) arena.release(g_off, g_bytes);
    g_bytes = 0;
    gplan = GridPlan{};
  }

  // CTAs for every request so that each ends within T; the small ones in bins.
  struct Share {
    std::vector<std::pair<Request*, int>> wide;  // request, CTAs
    std::vector<std::vector<Request*>> bins;     // one CTA each
  };
  static bool share(const std::vector<Request*>& rs, double T, int grid, Share& out) {
    out.wide.clear();
    out.bins.clear();
    std::vector<double> load;
    int used = 0;
    for (Request* r : rs) {  // longest first
      const double n = r->work_left(), one = n * r->seconds(1);
      if (r->least == 1 && one <= T) {
        size_t b = 0;
        while (b < load.size() && load[b] + one > T) ++b;
        if (b == load.size()) {
          load.push_back(0.0);
          out.bins.emplace_back();
        }
        load[b] += one;
        out.bins[b].push_back(r);
      } else {
        const double fixed = n * 6.5e-6, rest = n * (r->seconds(2) - 6.5e-6) * 2.0;
        if (T <= fixed) return false;
        const double c = std::ceil(rest / (T - fixed));
        if (c > grid) return false;
        const int ctas = std::max({(int)c, r->least, 2});
        out.wide.emplace_back(r, ctas);
        used += ctas;
      }
      if (used + (int)out.bins.size() > grid) return false;
    }
    return true;
  }

  // The small requests over all CTAs that the wide ones leave, the longest first to
  // the CTA with the least.
  static void spread(Share& out, int grid) {
    int used = 0;
    std::vector<std::pair<double, Request*>> rs;
    for (auto& w : out.wide) used += w.second;
    for (auto& b : out.bins)
      for (Request* r : b) rs.emplace_back(r->work_left() * r->seconds(1), r);
    const size_t n = std::min<size_t>(rs.size(), grid - used);
    if (n <= out.bins.size()) return;
    std::stable_sort(rs.begin(), rs.end(), [](const auto& a, const auto& b) { return a.first > b.first; });
    std::vector<double> load(n, 0.0);
    out.bins.assign(n, {});
    for (auto& r : rs) {
      const size_t b = std::min_element(load.begin(), load.end()) - load.begin();
      load[b] += r.first;
      out.bins[b].push_back(r.second);
    }
  }

  // Plans the running requests for the grid kernel. False when they do not fit it
  // together. (Not under the mutex: slots and arena are the worker's own, and cutting
  // the models takes milliseconds.)
  bool plan_grid(int32_t count) {
    drop_grid();
    std::vector<Request*> rs;
    int64_t nnz = 0, cols = 0;
    for (int32_t s = 0; s < count; ++s)
      if (slots[s]) {
        rs.push_back(slots[s]);
        nnz += slots[s]->model->nnz;
        cols += slots[s]->model->n_cols;
      }
    const int grid = bellman_grid();
    const bool f32 = !rs.empty() && rs[0]->model->lg32;
    for (const Request* r : rs)
      if ((r->model->lg32 != nullptr) != f32 || r->model->nnz >= kGridMostEntries) return false;
    // more requests than that would mostly follow one another on single CTAs, where
    // every CTA waits for the one with the most new requests (2000 requests/s, 360
    // running: 0.88e11 transition-updates/s shared, 0.89 to 0.96e11 per iteration)
    if (rs.empty() || (int)rs.size() > grid / 2) return false;
    size_t lists = 0;
    for (Request* r : rs) {
      if (r->least == 0) r->least = grid_least_ctas(r->model, r->fixed.data(), &r->columns);
      lists += r->columns * sizeof(GridMiss);
    }
    // no room for the lists of missed columns (most of the block below): the models
    // need not be cut to see it
    if (lists > arena.largest()) return false;
    std::stable_sort(rs.begin(), rs.end(), [](const Request* a, const Request* b) {
      return a->work_left() * a->seconds(1) > b->work_left() * b->seconds(1);
    });
    Share best, now;
    std::vector<GridCut> cuts;
    for (int attempt = 0;; ++attempt) {
      double hi = 0.0, lo = 0.0;
      for (const Request* r : rs) hi += r->work_left() * r->seconds(1);
      if (!share(rs, hi, grid, best)) return false;  // the least that the requests need is too much
      for (int i = 0; i < 20; ++i) {
        const double mid = 0.5 * (lo + hi);
        if (share(rs, mid, grid, now)) {
          hi = mid;
          std::swap(best, now);
        } else {
          lo = mid;
        }
      }
      // Two percent more time leave some of the wide requests' CTAs for the small ones,
      // which otherwise follow one another on as few as can be (20 of 5 ms arriving
      // beside one of 130: half of them done within 29 ms, within 4.9 so).
      if (!best.wide.empty() && !best.bins.empty() && share(rs, 1.02 * hi, grid, now)) std::swap(best, now);
      spread(best, grid);
      cuts.assign(rs.size(), GridCut{});
      bool ok = true;
      size_t i = 0;
      auto cut = [&](Request* r, int ctas) {
        if (!plan_grid_unit(r->model, r->fixed.data(), ctas, cuts[i++])) {
          r->least = ctas + std::max(1, ctas / 2);
          ok = false;
        }
      };
      for (auto& w : best.wide) cut(w.first, w.second);
      for (auto& b : best.bins) {
        // the one that ends first runs first
        std::stable_sort(b.begin(), b.end(), [](const Request* x, const Request* y) {
          return x->work_left() * x->seconds(1) < y->work_left() * y->seconds(1);
        });
        for (Request* r : b) cut(r, 1);
      }
      if (ok) break;
      if (attempt == 8) return false;
    }
    // units, and where their tables lie in the block
    g_units.clear();
    g_work.clear();
    g_reqs.clear();
    size_t at = 0, misses = 0, chunks = 0;
    auto take = [&](size_t bytes) {
      const size_t o = at;
      at += (bytes + 255) & ~size_t(255);
      return o;
    };
    int32_t steal_ctas = 0;
    bool copy = true;
    size_t need = 0, all = 0;
    auto unit = [&](Request* r, int first, int ctas) {
      const GridCut& c = cuts[g_units.size()];
      GridUnit u{};
      u.p = r->slot;
      u.n_chunks = (int32_t)c.win.size();
      u.one_window = c.one_window;
      u.first = first;
      u.ctas = ctas;
      u.single = r->model->n_cols == r->model->n_states ? 1 : 0;
      u.most_cols = c.most_cols;
      u.most_own = c.most_own;
      u.most_cells = c.most_cells;
      u.max_col = r->model->max_col;
      g_units.push_back(u);
      g_reqs.push_back(r);
      steal_ctas += ctas;
      chunks += c.chunk.size();
      misses += (size_t)ctas * c.most_cols;
      const size_t mine = grid_bytes(c, f32), with = mine + 64 + 20 * (size_t)c.entries;
      need = std::max(need, mine);
      all = std::max(all, with);
      copy = copy && with <= kResidentSmem;
    };
    int first = 0;
    for (auto& w : best.wide) {
      for (int c = 0; c < w.second; ++c) g_work.push_back(make_int2((int)g_units.size(), (int)g_units.size() + 1));
      unit(w.first, first, w.second);
      first += w.second;
    }
    for (auto& b : best.bins) {
      const int u0 = (int)g_units.size();
      for (Request* r : b) unit(r, first, 1);
      g_work.push_back(make_int2(u0, (int)g_units.size()));
      ++first;
    }
    const size_t n = g_units.size();
    const size_t o_units = take(n * sizeof(GridUnit)), o_work = take(g_work.size() * sizeof(int2)),
                 o_ctl = take(n * sizeof(StepControl)), o_steal = take(4 * sizeof(uint32_t) * (size_t)steal_ctas),
                 o_chunk = take(chunks * sizeof(int32_t)), o_win = take(chunks * sizeof(GridWindow)),
                 o_miss = take(misses * sizeof(GridMiss));
    size_t off;
    if (!arena.alloc(at, &off)) return false;  // no room in the budget: per-iteration launches
    g_off = off;
    g_bytes = at;
    unsigned char* block = base + off;
    gplan.units = d_gunits = (GridUnit*)(block + o_units);
    gplan.work = d_gwork = (int2*)(block + o_work);
    d_gctl = (StepControl*)(block + o_ctl);
    gplan.steal = (uint32_t*)(block + o_steal);
    gplan.steal_ctas = steal_ctas;
    gplan.grid = first;
    gplan.group = nnz >= 256 * cols || cols < 48 * (int64_t)first ? 32 : 8;
    gplan.f32 = f32 ? 1 : 0;
    gplan.smem = (uint32_t)((copy ? all : need) + 15) & ~15u;
    std::vector<int32_t> ch;
    std::vector<GridWindow> wn;
    ch.reserve(chunks);
    wn.reserve(chunks);
    GridMiss* miss = (GridMiss*)(block + o_miss);
    uint32_t* steal = gplan.steal;
    for (size_t i = 0; i < n; ++i) {
      GridUnit& u = g_units[i];
      const GridCut& c = cuts[i];
      u.chunk = (int32_t*)(block + o_chunk) + ch.size();
      u.win = (GridWindow*)(block + o_win) + wn.size();
      ch.insert(ch.end(), c.chunk.begin(), c.chunk.end());
      wn.insert(wn.end(), c.win.begin(), c.win.end());
      u.misses = miss;
      miss += (size_t)u.ctas * u.most_cols;
      u.steal = steal;
      steal += 4 * (size_t)u.ctas;
      u.ctl = d_gctl + i;
    }
    cudaError_t e = grid_prepare(gplan);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_gctl, 0, n * sizeof(StepControl), stream);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync((void*)g_units[0].chunk, ch.data(), ch.size() * sizeof(int32_t), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync((void*)g_units[0].win, wn.data(), wn.size() * sizeof(GridWindow), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);  // the host vectors go out of scope
    if (e != cudaSuccess) {
      cudaGetLastError();
      drop_grid();
      return false;
    }
    gplan.n_units = (int32_t)n;
    return true;
  }

  // Iterations of every unit in the next launch, about a quantum for each CTA;
  // returns the CTAs that still have work.
  int plan_quantum(std::vector<int2>& work) {
    work.assign(g_work.size(), make_int2(0, 0));
    std::vector<double> left(g_work.size(), 0.0);
    double longest = 0.0;
    auto per = [&](int u) { return g_reqs[u]->seconds(g_units[u].ctas); };
    for (size_t c = 0; c < g_work.size(); ++c) {
      for (int u = g_work[c].x; u < g_work[c].y; ++u)
        if (g_reqs[u]) left[c] += g_reqs[u]->work_left() * per(u);
      longest = std::max(longest, left[c]);
    }
    ++launch;
    int busy = 0;
    for (size_t c = 0; c < g_work.size(); ++c) {
      const int u0 = g_work[c].x, u1 = g_work[c].y;
      // CTAs with about as much left as the longest end with it; those with much less
      // run to their ends (they would take as long as it does)
      double budget = std::min(left[c], kQuantumSeconds);
      if (left[c] > 0.5 * longest && longest > kQuantumSeconds) budget = left[c] * (kQuantumSeconds / longest);
      int2& w = work[c];
      const auto give = [&](int u, double seconds) {
        const int32_t n = g_reqs[u]->iterations(seconds / per(u));
        g_units[u].iters = n;
        w = w.y == 0 ? make_int2(u, u + 1) : make_int2(std::min(w.x, u), std::max(w.y, u + 1));
        return Request::weighted(g_reqs[u]->k, n) * per(u);
      };
      if (u1 - u0 == 1) {  // its own CTAs
        if (g_reqs[u0]) give(u0, budget);
      } else {
        // Shortest work first gives the short ones their results early, but the work
        // of an infinite horizon is a guess that does not shrink: a few that converge
        // slowly would use up every launch. So when not all can run, a quarter of the
        // time goes to one request, another in every launch.
        for (int u = u0; u < u1; ++u) g_units[u].iters = 0;  // not in this launch
        if (left[c] > kQuantumSeconds) {
          int turn = u0 + (int)(launch % (uint64_t)(u1 - u0)), first = u0;
          while (!g_reqs[turn] && turn + 1 < u1) ++turn;
          while (!g_reqs[first] && first + 1 < u1) ++first;
          if (g_reqs[turn] && turn != first) budget -= give(turn, 0.25 * budget);
        }
        for (int u = u0; u < u1 && (w.y == 0 || budget > 1e-7); ++u)
          if (g_reqs[u] && g_units[u].iters == 0) budget -= give(u, budget);
      }
      busy += w.y > 0 ? 1 : 0;
    }
    return busy;
  }

  void retire(Request* r, const IterState& it) {
    const DevModel* m = r->model;
    const int32_t n = m->n_states;
    const int32_t k = it.done ? it.k_final : it.iter;
    unsigned char* p = base + r->off;
    auto step = [&](size_t x) { return (x + 255) & ~size_t(255); };
    uint64_t* V = (uint64_t*)p;
    double* out = (double*)(p + step(2 * (size_t)n * 8) + step(padded_u8(n)) + step(padded_i32(m->n_cols) * 4));
    r->result.resize(n);
    srv_export_kernel<<<std::min((n + 255) / 256, 1024), 256, 0, stream>>>(n, V + (size_t)(k & 1) * n, r->v_offset,
                                                                        r->v_scale, out);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(r->result.data(), out, sizeof(double) * n, cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    r->k = k;
    r->status = e != cudaSuccess ? cuda_status(e, "server retire") : (it.noconv ? IMDP_ENOCONV : IMDP_OK);
    r->finished = Clock::now();
    std::lock_guard<std::mutex> lk(mu);
    arena.release(r->off, r->bytes);
    for (Request*& g : g_reqs)
      if (g == r) g = nullptr;
    blocked = 0;
    slots[r->slot] = nullptr;
    std::memset(&probs_h[r->slot], 0, sizeof(Problem));
    r->slot = -1;
    r->done = true;
    cv.notify_all();
  }

  void run() {
    cudaSetDevice(device);
    std::vector<IterState> its;
    std::vector<StepControl> ctls;
    std::vector<int2> work;
    int32_t count = 0;  // slots [0, count) are in the launch
    bool stale = true;  // the per-iteration launches' tables are older than the slots
    bool refused = false;  // a shared launch did not fit the device
    bool fits = true;   // the running requests fit the grid kernel together, as far as known
    while (true) {
      bool changed = false;
      const Clock::time_point h0 = Clock::now();
      {
        std::unique_lock<std::mutex> lk(mu);
        bool any_active = false;
        for (Request* r : slots) any_active = any_active || r;
        if (!any_active && queue.empty()) {
          cv.wait_for(lk, std::chrono::milliseconds(50), [&] { return stop || !queue.empty(); });
        }
        if (stop) return;
        // admit in arrival order while a slot and budget are free
        while (!queue.empty()) {
          int slot = -1;
          for (int s = 0; s < max_active; ++s)
            if (!slots[s]) {
              slot = s;
              break;
            }
          if (slot < 0) break;
          Request* r = queue.front();
          if (!admit(r, slot)) {
            // the grid kernel's plan makes room, once for a request that then still has to wait
            if (!g_bytes || blocked == r->ticket) break;
            drop_grid();
            blocked = r->ticket;
            continue;
          }
          queue.pop_front();
          changed = true;
        }
      }
      int32_t hi = 0;
      for (int s = 0; s < max_active; ++s)
        if (slots[s]) hi = s + 1;
      if (hi == 0) continue;
      cudaError_t e = cudaSuccess;
      LaunchConfig lc;
      bool grid_kernel = false;
      if (changed || hi != count) {
        // slots without a request keep done = 1 (set at creation, kept on retire)
        stale = true;
        fits = fits || changed;
        count = hi;
        e = cudaMemcpyAsync(d_probs, probs_h.data(), sizeof(Problem) * count, cudaMemcpyHostToDevice, stream);
      }
      {
        std::lock_guard<std::mutex> lk(mu);
        lc = cfg;
      }
      if (lc.by_rule() && fits && !refused) {
        // planned again when a quarter of the CTAs have run out of work
        grid_kernel = gplan.n_units > 0 && !changed && plan_quantum(work) * 4 > gplan.grid * 3;
        if (!grid_kernel) {
          grid_kernel = fits = plan_grid(count);
          if (grid_kernel) plan_quantum(work);
        }
      }
      if (!grid_kernel) drop_grid();
      if (!grid_kernel && stale && e == cudaSuccess) {
        const imdp_status st = upload_tables(count);
        if (st != IMDP_OK) {
          std::lock_guard<std::mutex> lk(mu);
          fatal = st;
          for (Request* r : slots)
            if (r) {
              r->status = st;
              r->done = true;
            }
          cv.notify_all();
          return;
        }
        stale = false;
      }
      pending_host_ms = std::chrono::duration<double, std::milli>(Clock::now() - h0).count();
      StepLaunch L{};
      L.probs = d_probs;
      L.its = d_its;
      L.state_base = d_base;
      L.ctl = d_ctl;
      L.count = count;
      L.total_states = 0;
      L.any_infinite = 1;
      L.tiles = d_tiles;
      L.n_tiles = n_tiles;
      L.tile_cols = tile_cols;
      L.wide = d_wide;
      L.n_wide = n_wide;
      const int grid = bellman_grid();
      TraceRange trace("imdp server chunk");
      const Clock::time_point w0 = Clock::now();
      if (!ev0 && e == cudaSuccess) {
        e = cudaEventCreate(&ev0);
        if (e == cudaSuccess) e = cudaEventCreate(&ev1);
      }
      if (grid_kernel && e == cudaSuccess) {
        e = cudaMemcpyAsync(d_gunits, g_units.data(), sizeof(GridUnit) * g_units.size(), cudaMemcpyHostToDevice, stream);
        if (e == cudaSuccess)
          e = cudaMemcpyAsync(d_gwork, work.data(), sizeof(int2) * work.size(), cudaMemcpyHostToDevice, stream);
      }
      if (e == cudaSuccess) e = cudaEventRecord(ev0, stream);
      if (grid_kernel) {
        if (e == cudaSuccess) e = launch_bellman_grid(L, gplan, 0, stream);
        if (e == cudaErrorCooperativeLaunchTooLarge) {  // nothing was launched: per iteration from here on
          cudaGetLastError();
          refused = true;
          continue;
        }
      } else {
        for (int i = 0; i < chunk && e == cudaSuccess; ++i) e = launch_bellman_step(L, grid, stream, &side, &lc);
      }
      if (e == cudaSuccess) e = cudaEventRecord(ev1, stream);
      its.resize(count);
      StepControl c{};
      if (e == cudaSuccess) e = cudaMemcpyAsync(its.data(), d_its, sizeof(IterState) * count, cudaMemcpyDeviceToHost, stream);
      ctls.resize(grid_kernel ? g_units.size() : 0);
      if (e == cudaSuccess && !grid_kernel) e = cudaMemcpyAsync(&c, d_ctl, sizeof(c), cudaMemcpyDeviceToHost, stream);
      if (e == cudaSuccess && grid_kernel)
        e = cudaMemcpyAsync(ctls.data(), d_gctl, sizeof(StepControl) * ctls.size(), cudaMemcpyDeviceToHost, stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
      for (const StepControl& g : ctls) c.error |= g.error;
      if (e != cudaSuccess || c.error) {
        std::lock_guard<std::mutex> lk(mu);
        fatal = e != cudaSuccess ? cuda_status(e, "server step") : IMDP_ETIMEOUT;
        for (Request* r : slots)
          if (r) {
            r->status = fatal;
            r->done = true;
          }
        cv.notify_all();
        return;
      }
      float dev_ms = 0.f;
      cudaEventElapsedTime(&dev_ms, ev0, ev1);
      int active = 0;
      for (int s = 0; s < count; ++s) {
        Request* r = slots[s];
        active += r ? 1 : 0;
        if (r) r->k = its[s].iter;
        if (r && its[s].done) {
          retire(r, its[s]);
          fits = true;
        }
      }
      {
        std::lock_guard<std::mutex> lk(mu);
        st_device_ms += dev_ms;
        st_chunks += 1;
        st_shared += grid_kernel ? 1 : 0;
        st_slots += active;
        // wall time from this chunk's launches to the end of its retirements;
        // admission and table uploads before the next chunk are added there
        st_wall_ms += std::chrono::duration<double, std::milli>(Clock::now() - w0).count() + pending_host_ms;
      }
      pending_host_ms = 0.0;
    }
  }
  double pending_host_ms = 0.0;  // admission and table work before the next chunk (worker only)

  static uint64_t eps_fixed(double eps) {
    if (eps >= 1.0) return kOne + 1;
    const double x = eps * 9223372036854775808.0;
    uint64_t f = (uint64_t)x;
    if ((double)f < x) f += 1;
    return f;
  }
};

}  // namespace imdp

using namespace imdp;

struct imdp_server {
  Server* s;
};

extern "C" {

imdp_status imdp_server_stats(imdp_server* srv, double* device_ms, double* wall_ms, int64_t* chunks,
                              double* mean_requests) {
  set_error("");
  if (!srv || !srv->s) { set_error("NULL server"); return IMDP_EINVAL; }
  Server* S = srv->s;
  std::lock_guard<std::mutex> lk(S->mu);
  if (device_ms) *device_ms = S->st_device_ms;
  if (wall_ms) *wall_ms = S->st_wall_ms;
  if (chunks) *chunks = S->st_chunks;
  if (mean_requests) *mean_requests = S->st_chunks ? S->st_slots / (double)S->st_chunks : 0.0;
  return IMDP_OK;
}

imdp_status imdp_server_launches(imdp_server* srv, int64_t* shared, int64_t* per_iteration) {
  set_error("");
  if (!srv || !srv->s) { set_error("NULL server"); return IMDP_EINVAL; }
  Server* S = srv->s;
  std::lock_guard<std::mutex> lk(S->mu);
  if (shared) *shared = S->st_shared;
  if (per_iteration) *per_iteration = (S->st_chunks - S->st_shared) * S->chunk;
  return IMDP_OK;
}

imdp_status imdp_server_set_launch(imdp_server* srv, const imdp_launch_config* cfg) {
  set_error("");
  if (!srv || !srv->s || !cfg) { set_error("NULL server or configuration"); return IMDP_EINVAL; }
  if (cfg->kernel < 0 || cfg->kernel > 2 || cfg->tile_entries < 0 || cfg->wide_col < 0) {
    set_error("bad launch configuration");
    return IMDP_EINVAL;
  }
  LaunchConfig c;
  c.kernel = cfg->kernel;
  c.cta_warps = cfg->cta_warps;
  c.ctas_per_sm = cfg->ctas_per_sm;
  c.tile_entries = cfg->tile_entries;
  c.wide_col = cfg->wide_col;
  std::lock_guard<std::mutex> lk(srv->s->mu);
  srv->s->cfg = c;  // requests admitted from now on are planned with its limits
  return IMDP_OK;
}

imdp_status imdp_server_create(size_t hbm_budget, imdp_server** out) {
  set_error("");
  if (!out || hbm_budget < (size_t(1) << 20)) { set_error("server needs out and a budget of at least 1 MiB"); return IMDP_EINVAL; }
  *out = nullptr;
  int n = 0;
  if (cudaGetDeviceCount(&n) != cudaSuccess || n == 0) {
    cudaGetLastError();
    set_error("no CUDA device");
    return IMDP_EDEVICE;
  }
  Server* S = new Server(hbm_budget);
  cudaGetDevice(&S->device);
  S->slots.assign(S->max_active, nullptr);
  S->probs_h.assign(S->max_active, Problem{});
  cudaError_t e = cudaStreamCreateWithFlags(&S->stream, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = S->side.create();
  if (e == cudaSuccess) e = cudaMalloc(&S->base, S->arena.size());
  if (e == cudaSuccess) e = cudaMalloc(&S->d_probs, sizeof(Problem) * S->max_active);
  if (e == cudaSuccess) e = cudaMalloc(&S->d_its, sizeof(IterState) * S->max_active);
  if (e == cudaSuccess) e = cudaMalloc(&S->d_ctl, sizeof(StepControl));
  if (e == cudaSuccess) e = cudaMalloc(&S->d_base, sizeof(int32_t) * 2);
  if (e == cudaSuccess) e = cudaMemset(S->d_ctl, 0, sizeof(StepControl));
  if (e == cudaSuccess) e = cudaMemset(S->d_base, 0, sizeof(int32_t) * 2);
  if (e == cudaSuccess) e = cudaMemset(S->d_probs, 0, sizeof(Problem) * S->max_active);
  if (e != cudaSuccess) {
    const imdp_status st = cuda_status(e, "server create");
    delete S;
    return st;
  }
  // every slot starts "done" (empty)
  std::vector<IterState> init(S->max_active);
  for (auto& it : init) {
    std::memset(&it, 0, sizeof(it));
    it.done = 1;
  }
  e = cudaMemcpy(S->d_its, init.data(), sizeof(IterState) * S->max_active, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    const imdp_status st = cuda_status(e, "server create");
    delete S;
    return st;
  }
  S->worker = std::thread([S] { S->run(); });
  *out = new imdp_server{S};
  return IMDP_OK;
}

imdp_status imdp_server_submit(imdp_server* srv, imdp_model* m, const imdp_spec* spec, uint64_t* ticket) {
  set_error("");
  if (!srv || !m || !spec || !ticket) { set_error("NULL argument"); return IMDP_EINVAL; }
  Server* S = srv->s;
  if (m->device != S->device) { set_error("model and server must be on one device"); return IMDP_EINVAL; }
  if (is_slice(m->dev)) { set_error("slices of a state-sharded model run in sessions only"); return IMDP_EINVAL; }
  imdp_status st = check_spec(m->dev, spec);
  if (st != IMDP_OK) return st;
  Request* r = new Request();
  r->model = m->dev;
  r->spec = *spec;
  if (spec->n_reach > 0) r->reach.assign(spec->reach, spec->reach + spec->n_reach);
  if (spec->property == IMDP_REACH_AVOID && spec->n_avoid > 0) r->avoid.assign(spec->avoid, spec->avoid + spec->n_avoid);
  if (spec->property == IMDP_REWARD) r->reward.assign(spec->reward, spec->reward + m->dev->n_states);
  for (int32_t v : r->avoid)
    if (std::find(r->reach.begin(), r->reach.end(), v) != r->reach.end()) {
      delete r;
      set_error("a state is in both the reach and the avoid set");
      return IMDP_EINVAL;
    }
  r->spec.reach = nullptr;
  r->spec.avoid = nullptr;
  r->spec.reward = nullptr;
  r->bytes = working_bytes(m->dev, spec);
  if (r->bytes > S->arena.size()) {
    delete r;
    set_error("request needs more device memory than the server's budget");
    return IMDP_ENOMEM;
  }
  std::lock_guard<std::mutex> lk(S->mu);
  if (S->fatal != IMDP_OK) {
    delete r;
    set_error("server stopped after a device error");
    return S->fatal;
  }
  if (S->queue.size() >= 1000000) {
    delete r;
    set_error("server queue full");
    return IMDP_EBUSY;
  }
  r->ticket = S->next_ticket++;
  r->submitted = Clock::now();
  S->queue.push_back(r);
  S->all[r->ticket] = r;
  *ticket = r->ticket;
  S->cv.notify_all();
  return IMDP_OK;
}

imdp_status imdp_server_poll(imdp_server* srv, uint64_t ticket, double* V_out, int32_t* k_out, double* latency_ms) {
  if (!srv) { set_error("NULL server"); return IMDP_EINVAL; }
  Server* S = srv->s;
  std::lock_guard<std::mutex> lk(S->mu);
  auto it = S->all.find(ticket);
  if (it == S->all.end()) { set_error("unknown ticket"); return IMDP_ENOTFOUND; }
  Request* r = it->second;
  if (!r->done) return IMDP_EPENDING;
  const imdp_status st = r->status;
  if (st == IMDP_OK || st == IMDP_ENOCONV) {
    if (V_out) {
      if (is_device_pointer(V_out)) {
        cudaMemcpy(V_out, r->result.data(), sizeof(double) * r->result.size(), cudaMemcpyHostToDevice);
      } else {
        std::memcpy(V_out, r->result.data(), sizeof(double) * r->result.size());
      }
    }
    if (k_out) *k_out = r->k;
    if (latency_ms) *latency_ms = std::chrono::duration<double, std::milli>(r->finished - r->submitted).count();
  }
  S->all.erase(it);
  delete r;
  return st;
}

imdp_status imdp_server_wait(imdp_server* srv, uint64_t ticket, double timeout_ms, double* V_out, int32_t* k_out,
                             double* latency_ms) {
  if (!srv) { set_error("NULL server"); return IMDP_EINVAL; }
  Server* S = srv->s;
  {
    std::unique_lock<std::mutex> lk(S->mu);
    auto it = S->all.find(ticket);
    if (it == S->all.end()) { set_error("unknown ticket"); return IMDP_ENOTFOUND; }
    Request* r = it->second;
    const bool ok = S->cv.wait_for(lk, std::chrono::duration<double, std::milli>(timeout_ms), [&] { return r->done; });
    if (!ok) { set_error("timed out waiting for the request"); return IMDP_ETIMEOUT; }
  }
  return imdp_server_poll(srv, ticket, V_out, k_out, latency_ms);
}

void imdp_server_destroy(imdp_server* srv) {
  if (!srv) return;
  delete srv->s;
  delete srv;
}

}  // extern "C"
