// Resident solver sessions: device state of value iteration (Eq. 2) for a batch
// of problems, the iteration driver (graph-captured chunks of Bellman steps)
// and the export of (V, k, residual, policy) as value_iteration returns them
// (Sec. 3.2).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include <cuda_runtime.h>

#include "imdp_internal.h"

namespace imdp {

namespace {

__global__ void init_values_kernel(int64_t n, const uint8_t* __restrict__ fixed, uint64_t* __restrict__ V0) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    V0[i] = fixed[i] == 1 ? kOne : 0ull;
}

// W (Q1.63) -> V = offset + scale * W in binary64; with `prev`, writes
// scale * (W - prev), the Bellman residual V_k - V_{k-1}.
__global__ void export_values_kernel(int32_t n, const uint64_t* __restrict__ V, const uint64_t* __restrict__ prev,
                                     double offset, double scale_v, double* __restrict__ out) {
  const double scale = scale_v / 9223372036854775808.0;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (prev) {
      const uint64_t a = V[i], b = prev[i];
      out[i] = a >= b ? (double)(a - b) * scale : -(double)(b - a) * scale;
    } else {
      out[i] = offset + (double)V[i] * scale;
    }
  }
}


__global__ void fill_i32_kernel(int64_t n, int32_t* p, int32_t v) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = v;
}

// eps in Q1.63 rounded up, so an integer residual r satisfies r < eps_fix
// exactly when r * 2^-63 < eps.
uint64_t eps_to_fixed(double eps) {
  if (eps >= 1.0) return kOne + 1;
  const double x = eps * 9223372036854775808.0;
  uint64_t f = (uint64_t)x;
  if ((double)f < x) f += 1;
  return f;
}

constexpr int kGraphChunk = 16;

// One problem's values in read_all: its words, and where they go.
struct ExportItem {
  const uint64_t* V;
  double* out;
  double offset, scale;
  int32_t n;
};

// The values of many problems, a row of blocks for each.
__global__ void export_batch_kernel(const ExportItem* __restrict__ items) {
  const ExportItem it = items[blockIdx.y];
  const double scale = it.scale / 9223372036854775808.0;
  for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < it.n; i += gridDim.x * blockDim.x)
    it.out[i] = it.offset + (double)it.V[i] * scale;
}

}  // namespace

// Affine map of a reward problem into [0, 1] (V = lo + D W). Rewards r, discount
// g, horizon K: if V_{k-1} lies in [a, b], the averaging operator keeps
// T(V_{k-1}) in [a, b], so V_k = r + g T(V_{k-1}) lies in [rmin + g a, rmax + g b];
// from V_0 = r this gives V_k in [rmin A_k, rmax A_k] with A_k = sum_{i<=k} g^i,
// and every V_k, k <= K, lies in [min(rmin, rmin A), max(rmax, rmax A)].
void reward_map(const double* r, int32_t n, double g, int32_t K, bool infinite, double* lo, double* D) {
  double rmin = r[0], rmax = r[0];
  for (int32_t s = 1; s < n; ++s) {
    rmin = r[s] < rmin ? r[s] : rmin;
    rmax = r[s] > rmax ? r[s] : rmax;
  }
  double A;
  if (infinite) A = 1.0 / (1.0 - g);
  else if (g == 1.0) A = (double)K + 1.0;
  else A = (1.0 - std::pow(g, (double)K + 1.0)) / (1.0 - g);
  const double a = std::min(rmin, rmin * A), b = std::max(rmax, rmax * A);
  // widen by a relative margin so rounding never pushes W outside [0, 1]
  const double span = b - a, pad = 1e-9 * (span > 0 ? span : 1.0) + 1e-300;
  *lo = a - pad;
  *D = (span > 0 ? span : 1.0) + 2 * pad;
}

imdp_status check_spec(const DevModel* m, const imdp_spec* sp) {
  if (!sp) { set_error("spec is NULL"); return IMDP_EINVAL; }
  if (sp->property != IMDP_REACH && sp->property != IMDP_REACH_AVOID && sp->property != IMDP_REWARD) {
    set_error("unknown property"); return IMDP_EINVAL;
  }
  if (sp->property == IMDP_REWARD) {
    // Sec. 3.2: rewards per state, discount in (0, 1] (strictly below 1 for an infinite horizon)
    if (!sp->reward) { set_error("reward property needs a reward vector"); return IMDP_EINVAL; }
    if (!(sp->discount > 0.0) || !(sp->discount <= 1.0) || (sp->infinite_time && !(sp->discount < 1.0))) {
      set_error("discount must be in (0, 1] (finite horizon) or (0, 1) (infinite horizon)"); return IMDP_EINVAL;
    }
    for (int32_t s = 0; s < m->n_states; ++s)
      if (!(sp->reward[s] == sp->reward[s]) || sp->reward[s] > 1e300 || sp->reward[s] < -1e300) {
        set_error("rewards must be finite"); return IMDP_EINVAL;
      }
  }
  if (sp->horizon < 0) { set_error("horizon must be >= 0"); return IMDP_EINVAL; }
  if (sp->infinite_time && !(sp->eps > 0.0)) { set_error("eps must be > 0 for an infinite horizon"); return IMDP_EINVAL; }
  if (sp->n_reach < 0 || (sp->n_reach > 0 && !sp->reach)) { set_error("bad reach set"); return IMDP_EINVAL; }
  if (sp->property == IMDP_REACH_AVOID && (sp->n_avoid < 0 || (sp->n_avoid > 0 && !sp->avoid))) {
    set_error("bad avoid set"); return IMDP_EINVAL;
  }
  for (int32_t i = 0; i < sp->n_reach; ++i)
    if (sp->reach[i] < 0 || sp->reach[i] >= m->n_states) { set_error("reach state out of range"); return IMDP_EINVAL; }
  if (sp->property == IMDP_REACH_AVOID)
    for (int32_t i = 0; i < sp->n_avoid; ++i)
      if (sp->avoid[i] < 0 || sp->avoid[i] >= m->n_states) { set_error("avoid state out of range"); return IMDP_EINVAL; }
  return IMDP_OK;
}

Session::~Session() {
  if (graph) cudaGraphExecDestroy(graph);
  side.destroy();
}

void* Session::get_memory(size_t bytes) {
  void* p = nullptr;
  if (cudaMalloc(&p, bytes) == cudaSuccess) return p;
  cudaGetLastError();
  return nullptr;
}

void Session::put_memory(void* p) { cudaFree(p); }

imdp_status Session::create(const std::vector<DevModel*>& ms, const std::vector<const imdp_spec*>& specs,
                            const int32_t* want_policy, cudaStream_t st, Session** out) {
  *out = nullptr;
  const int count = (int)ms.size();
  for (int p = 0; p < count; ++p) {
    imdp_status s = check_spec(ms[p], specs[p]);
    if (s != IMDP_OK) return s;
  }
  Session* S = new Session();
  S->count = count;
  S->models = ms;
  cudaGetDevice(&S->device);
  S->base_h.assign(count + 1, 0);
  for (int p = 0; p < count; ++p) S->base_h[p + 1] = S->base_h[p] + ms[p]->n_states;
  const int64_t total = S->base_h[count];
  if (total >= (int64_t(1) << 31)) { delete S; set_error("batch too large"); return IMDP_EINVAL; }
  S->total = total;
  std::vector<uint8_t> fixed((size_t)total, 0);
  for (int p = 0; p < count; ++p) {
    const imdp_spec* sp = specs[p];
    uint8_t* f = fixed.data() + S->base_h[p];
    if (sp->property != IMDP_REWARD)
      for (int32_t i = 0; i < sp->n_reach; ++i) f[sp->reach[i]] = 1;
    if (sp->property == IMDP_REACH_AVOID)
      for (int32_t i = 0; i < sp->n_avoid; ++i) {
        if (f[sp->avoid[i]] == 1) { delete S; set_error("a state is in both the reach and the avoid set"); return IMDP_EINVAL; }
        f[sp->avoid[i]] = 2;
      }
  }
  S->v_offset.assign(count, 0.0);
  S->v_scale.assign(count, 1.0);
  S->w0.assign(count, nullptr);
  // rank problems by horizon, longest first (infinite horizons first of all):
  // tiles laid out in this order leave the finished problems' tiles at the end
  S->order.resize(count);
  for (int p = 0; p < count; ++p) S->order[p] = p;
  std::stable_sort(S->order.begin(), S->order.end(), [&](int a, int b) {
    const int64_t ka = specs[a]->infinite_time ? INT64_MAX : specs[a]->horizon;
    const int64_t kb = specs[b]->infinite_time ? INT64_MAX : specs[b]->horizon;
    return ka > kb;
  });
  S->fixed_h = fixed;
  S->rank_of = S->alloc<int32_t>(count);
  S->rank_tile_end = S->alloc<int32_t>(count);
  // each problem's hint block starts on a 16-byte boundary and is padded, so
  // the kernel's bulk copies of hint windows stay aligned and in bounds
  for (int p = 0; p < count; ++p) S->total_cols += (int64_t)padded_i32(ms[p]->n_cols);
  S->hints = S->alloc<int32_t>((size_t)S->total_cols);
  S->fixed = S->alloc<uint8_t>(padded_u8(total));
  S->V = S->alloc<uint64_t>(2 * total);
  S->base = S->alloc<int32_t>(count + 1);
  S->probs = S->alloc<Problem>(count);
  S->its = S->alloc<IterState>(count);
  S->ctl = S->alloc<StepControl>(1);
  if (!S->hints || !S->fixed || !S->V || !S->base || !S->probs || !S->its || !S->ctl || !S->rank_of ||
      !S->rank_tile_end) {
    delete S; set_error("device allocation failed (session)"); return IMDP_ENOMEM;
  }
  S->probs_h.resize(count);
  S->policy_cells.assign(count, 0);
  int64_t col_off = 0;
  for (int p = 0; p < count; ++p) {
    DevModel* m = ms[p];
    const imdp_spec* sp = specs[p];
    Problem& P = S->probs_h[p];
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
    P.fixed = S->fixed + S->base_h[p];
    P.hint = S->hints + col_off;
    col_off += (int64_t)padded_i32(m->n_cols);
    P.V[0] = S->V + S->base_h[p];
    P.V[1] = S->V + total + S->base_h[p];
    P.n_states = m->n_states;
    P.pessimistic = sp->pessimistic ? 1 : 0;
    P.maximize = sp->maximize ? 1 : 0;
    P.property = sp->property;
    P.infinite = sp->infinite_time ? 1 : 0;
    // a slice holds part of the states: its own residual decides nothing, the
    // caller stops it on the residual of all slices (imdp_session_residual)
    P.external_stop = (P.infinite && is_slice(m)) ? 1 : 0;
    P.horizon = sp->infinite_time ? (sp->horizon > 0 ? sp->horizon : 1000000) : sp->horizon;
    P.eps_fix = sp->infinite_time ? eps_to_fixed(sp->eps) : 0;
    if (sp->property == IMDP_REWARD) {
      const int32_t n = m->n_states;
      double lo, D;
      reward_map(sp->reward, n, sp->discount, P.horizon, P.infinite != 0, &lo, &D);
      S->v_offset[p] = lo;
      S->v_scale[p] = D;
      std::vector<int64_t> c(n);
      std::vector<uint64_t> w(n);
      const double g = sp->discount;
      for (int32_t s = 0; s < n; ++s) {
        // W_k = c_s + g T(W_{k-1}),  c_s = (r_s - lo (1 - g)) / D  (signed Q2.62)
        const double cs = (sp->reward[s] - lo * (1.0 - g)) / D;
        c[s] = (int64_t)std::llround(cs * 4611686018427387904.0);
        const double ws = std::min(1.0, std::max(0.0, (sp->reward[s] - lo) / D));
        w[s] = (uint64_t)std::llround(ws * 4611686018427387904.0) << 1;
        if (m->lg32) w[s] = round_value32(w[s]);  // values of 32-bit storage keep 32 bits
      }
      int64_t* d_c = S->alloc<int64_t>(n);
      uint64_t* d_w = S->alloc<uint64_t>(n);
      if (!d_c || !d_w) { delete S; set_error("device allocation failed (reward)"); return IMDP_ENOMEM; }
      cudaError_t er = cudaMemcpyAsync(d_c, c.data(), sizeof(int64_t) * n, cudaMemcpyHostToDevice, st);
      if (er == cudaSuccess) er = cudaMemcpyAsync(d_w, w.data(), sizeof(uint64_t) * n, cudaMemcpyHostToDevice, st);
      if (er == cudaSuccess) er = cudaStreamSynchronize(st);
      if (er != cudaSuccess) { delete S; return cuda_status(er, "reward setup"); }
      P.rbias = d_c;
      S->w0[p] = d_w;
      P.gamma_fix = g >= 1.0 ? kOne : (uint64_t)std::llround(g * 9223372036854775808.0);
      if (P.infinite) P.eps_fix = eps_to_fixed(sp->eps / D);
    }
    S->max_horizon = std::max(S->max_horizon, P.horizon);
    S->any_infinite = S->any_infinite || P.infinite;
    if (want_policy && want_policy[p]) {
      const size_t cells = (size_t)(P.infinite ? 1 : P.horizon) * m->n_states;
      P.policy = S->alloc<int32_t>(cells);
      if (!P.policy) { delete S; set_error("device allocation failed (policy)"); return IMDP_ENOMEM; }
      P.policy_mode = P.infinite ? 2 : 1;
      S->policy_cells[p] = (int64_t)cells;
    }
  }
  cudaError_t e = cudaMemsetAsync(S->fixed, 0, padded_u8(total), st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(S->fixed, fixed.data(), total, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(S->base, S->base_h.data(), sizeof(int32_t) * (count + 1), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(S->probs, S->probs_h.data(), sizeof(Problem) * count, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // host staging vectors go out of scope
  if (e != cudaSuccess) { delete S; return cuda_status(e, "session setup"); }
  S->L.probs = S->probs;
  S->L.its = S->its;
  S->L.state_base = S->base;
  S->L.ctl = S->ctl;
  S->L.count = count;
  S->L.total_states = (int32_t)total;
  S->L.any_infinite = S->any_infinite ? 1 : 0;
  if (count == 1 && !is_slice(ms[0]) && ms[0]->n_states <= kTinyMaxStates && ms[0]->n_cols <= kTinyMaxCols &&
      ms[0]->nnz <= kTinyMaxEntries) {
    S->L.tiny_ok = 1;
    S->L.tiny_states = ms[0]->n_states;
    S->L.tiny_cols = ms[0]->n_cols;
    S->L.tiny_entries = (int32_t)ms[0]->nnz;
  }
  // the kernel by rule for this batch's shape: long columns (the mean over
  // all problems) the direct kernel; short ones the slice kernel when every
  // model already carries its slice layout (building one costs about as much as
  // 450 iterations of the slice kernel save on the pendulum shape), else ring
  {
    int64_t nnz = 0, cols = 0;
    bool all32 = true, laid_out = true;
    for (DevModel* m : ms) {
      nnz += m->nnz;
      cols += m->n_cols;
      all32 = all32 && m->lg32 != nullptr;
      std::lock_guard<std::mutex> lk(m->slices_mu);
      laid_out = laid_out && m->slices != nullptr;
    }
    if (nnz >= kRuleLongColumn * std::max<int64_t>(cols, 1))
      S->L.shape_rule = kKernelDirect;
    else if (laid_out)
      S->L.shape_rule = kKernelSlice;
    S->L.shape_f32 = all32 ? 1 : 0;
  }
  S->grid = bellman_grid();
  imdp_status r = S->plan_resident(specs, true, st);
  if (r == IMDP_OK) r = S->plan_grid(st);
  // (left to the grid kernel, whose shares do not fit)
  if (r == IMDP_OK && !S->plans_long_steps() && S->grid_possible()) r = S->plan_resident(specs, false, st);
  if (r != IMDP_OK) { delete S; return r; }
  const bool slice = resolve_launch(S->L, &S->cfg).kernel == kKernelSlice;
  r = slice ? S->prepare_slices(st) : IMDP_OK;
  if (r != IMDP_OK) { delete S; return r; }
  std::vector<Tile> tiles;
  std::vector<int2> wide;
  S->build_plan(S->cfg, tiles, wide);
  r = S->install_plan(tiles, wide, st, slice);
  if (r != IMDP_OK) { delete S; return r; }
  r = S->reset(st);
  if (r != IMDP_OK) { delete S; return r; }
  *out = S;
  return IMDP_OK;
}

bool Session::grid_possible() const {
  const DevModel* m = models[0];
  if (L.tiny_ok || count != 1 || is_slice(m) || m->nnz >= kGridMostEntries) return false;
  // Many long columns stay on the direct kernel: it settles a missed column while
  // its entries are still in L1 and L2 (100 iterations, direct and grid kernel, ms:
  // 48,000 columns of 500 entries 21.0 / 19.1, 56,000 of 376 16.7 / 16.5, 84,000 of
  // 376 20.2 / 20.8; on 32-bit storage 42,000 of 376 8.2 / 7.0, 48,000 of 500 15.7 /
  // 15.9, 90,000 of 300 14.5 / 16.4). Against the ring kernel, which short columns
  // take otherwise, it gains at any number (126,000 of 230 20.5 / 17.5).
  // So do very long columns for few iterations: in the first ones nearly all of them
  // are settled, which the block-wide kernel does faster (3,841 columns of 2,228
  // entries, direct and block-wide / grid kernel, ms: 32 iterations 4.3 / 5.1, 64 6.4 /
  // 6.5, 100 8.3 / 7.8; 3,001 of 1,800 16 iterations 1.77 / 1.93, 32 3.13 / 3.06). On
  // 32-bit storage that keeps most of them exact the stream has two kinds of columns
  // and gains less (3,841 of 2,228 100 iterations 8.5 / 9.3, 200 14.0 / 14.4; 7,681 of
  // them 14.4 / 14.6 and 24.0 / 22.8; 5,001 of 2,000 100 iterations 10.4 / 10.9; 3,001
  // of 1,800 100 iterations 6.0 / 5.8).
  const double k = (double)m->nnz / std::max(m->n_cols, 1);
  int32_t least = k >= 2000 ? 64 : (k >= 1500 ? 32 : 0);
  if (m->lg32 && k >= 2000 && m->exact_entries >= 0.5 * m->nnz) least = m->n_cols <= 4500 ? INT32_MAX : 128;
  if (least == INT32_MAX || (!any_infinite && max_horizon < least)) return false;
  return m->nnz < (int64_t)kRuleLongColumn * m->n_cols || m->n_cols <= (m->lg32 ? 45000 : 56000);
}

imdp_status Session::plan_resident(const std::vector<const imdp_spec*>& specs, bool beside_grid, cudaStream_t st) {
  resident = ResidentPlan{};
  bool any32 = false, any64 = false;
  for (const DevModel* m : models) {
    if (is_slice(m)) return IMDP_OK;
    (m->lg32 ? any32 : any64) = true;
  }
  if (any32 && any64) return IMDP_OK;
  const bool f32 = any32;
  // units: the problems, or the parts of one finite-horizon problem (small
  // neighbours together, so that a CTA's warps have columns enough)
  struct Work {
    ResidentUnit u;
    int64_t entries, work;
  };
  std::vector<Work> us;
  auto entries_of = [&](const DevModel* m, int32_t a, int32_t b) {
    return (int64_t)m->h_colptr[m->h_stateptr[b]] - m->h_colptr[m->h_stateptr[a]];
  };
  const bool parts = count == 1 && !specs[0]->infinite_time && models[0]->h_parts.size() > 2;
  if (parts) {
    const DevModel* m = models[0];
    const std::vector<int32_t>& b = m->h_parts;
    // Columns of a unit, at least: small neighbours go together. A state or two
    // detached from a model (an absorbing state of its own) would otherwise count
    // like the model itself (200 iterations of 5 states and one more: 0.29 ms as two
    // units, 0.26 as one; of 240 and one more 0.65, 0.60).
    int32_t largest = 0;
    for (size_t i = 0; i + 1 < b.size(); ++i)
      largest = std::max(largest, m->h_stateptr[b[i + 1]] - m->h_stateptr[b[i]]);
    const int64_t least = std::min(192, std::max({7, m->n_cols / (8 * grid), largest / 8}));
    const auto columns = [&](int32_t s0, int32_t s1) { return (int64_t)m->h_stateptr[s1] - m->h_stateptr[s0]; };
    for (size_t i = 0; i + 1 < b.size();) {
      size_t j = i + 1;
      while (j + 1 < b.size() && columns(b[i], b[j]) < least) ++j;
      // what is left at the end goes to the unit before
      const bool rest = !us.empty() && columns(b[i], b[j]) < least;
      if (!rest) us.push_back(Work{ResidentUnit{0, b[i], b[j]}, 0, 0});
      Work& w = us.back();
      w.u.s1 = b[j];
      w.work = w.entries = entries_of(m, w.u.s0, w.u.s1);
      i = j;
    }
  } else {
    for (int p = 0; p < count; ++p) {
      const int64_t e = entries_of(models[p], 0, models[p]->n_states);
      const int64_t K = specs[p]->infinite_time ? 1000 : specs[p]->horizon;
      us.push_back(Work{ResidentUnit{p, 0, models[p]->n_states}, e, e * std::max<int64_t>(K, 1)});
    }
  }
  int64_t entries = 0, work = 0, most = 0, cols = 0, longest = 1;  // iterations of the longest (parts: 1)
  int32_t states = 0, max_col = 0;
  for (const Work& w : us) {
    longest = std::max(longest, w.work / std::max<int64_t>(w.entries, 1));
    entries += w.entries;
    work += w.work;
    most = std::max(most, w.work);
    states = std::max(states, w.u.s1 - w.u.s0);
  }
  resident.single = 1;
  for (const DevModel* m : models) {
    max_col = std::max(max_col, m->max_col);
    cols += m->n_cols;
    resident.single = resident.single && m->n_cols == m->n_states;
  }
  // The very smallest stay on the single-CTA kernel, which has less to set up: up to 5
  // states of one action (200 iterations of 5: 212 us, 232 here; of 9 columns 325 and
  // 238), and with the residual of an infinite horizon up to 5 states of 16 columns
  // (64 iterations of 3 states and 3 columns 127 and 165 us, 72 of 5 and 15 232 and 277).
  if (L.tiny_ok && states <= 5 && cols <= (any_infinite ? 16 : (resident.single ? 5 : 0))) return IMDP_OK;
  const int32_t n_units = (int32_t)us.size();
  std::stable_sort(us.begin(), us.end(), [](const Work& a, const Work& b) { return a.work > b.work; });
  // Cluster size. More CTAs to a unit cost synchronisation; fewer leave the GPU
  // idle (too few units), end on one long unit (uneven work), or keep so much in
  // progress that it no longer sits in L2. Measured (64-bit storage, ms): 4096
  // parts of 0.5 MB 66 / 69 / 96 with 1 / 2 / 4 CTAs; 256 problems of 5 MB on
  // average with horizons from 100 to 500 82 / 88 / 98 with 4 / 6 / 8.
  const double unit_bytes = (double)entries / n_units * (f32 ? 12.0 : 20.0);
  int c = 1;
  while (c < kMaxCluster && ((int64_t)n_units * c < grid || unit_bytes * (grid / c) > 200e6 ||
                             (double)most / c > 1.7 * (double)work / grid))
    c *= 2;
  // Small units: at least 7 columns to a CTA (200 iterations of 12 columns 276 us
  // with one CTA, 310 with 4; 20 columns 330 with 2 or 4; 200 columns of 12 entries
  // 690 / 525 / 457 with 1 / 2 / 16).
  while (c > 1 && cols < 7 * (int64_t)c * n_units) c /= 2;
  const bool alone = count == 1 && n_units == 1;
  // Two CTAs of an SM overlap each other's barriers while both their units stay
  // in L2 (4096 parts of 0.3 MB on 32-bit storage: 68 ms against 74 with one) and
  // have room beside each other (below).
  const auto two_of = [&](int c) { return n_units * (int64_t)c >= 2 * grid && unit_bytes * (2 * grid / c) <= 100e6; };
  // Half the warps also where they hold a CTA's few short columns: their barriers
  // are cheaper (5 columns 238 us against 251, 600 columns 607 against 799).
  const bool few = alone && cols <= 48 * c && entries <= 32 * cols;
  // Seconds for all iterations: per-iteration launches take about 10 us each and
  // 0.64 transitions a cycle and SM, this kernel about 3 us and 1.17 on the SMs it
  // covers, the grid kernel (one problem only) about 6.5 us and 1 on all.
  const double hz = 1.9e9, iters = (double)longest, all_work = (double)work;
  double other = iters * 10e-6 + all_work / (0.64 * grid * hz);
  const double by_grid = iters * 6.5e-6 + all_work / (1.0 * grid * hz);
  if (beside_grid && grid_possible()) other = std::min(other, by_grid);
  const auto spread = [&](int c) {
    return iters * 3e-6 + all_work / (1.17 * std::min<double>(grid, (double)n_units * c) * hz);
  };
  if (spread(c) > other) return IMDP_OK;
  // Ranks of a unit: contiguous states of about equal work. False when a rank's
  // share does not fit a CTA.
  std::vector<int32_t> bounds;
  const auto shape = [&](int c) -> bool {
    int64_t rank_entries = 0;
    const bool two = two_of(c);
    resident.threads = two || few ? kResidentThreads / 2 : kResidentThreads;
    if (resident_bytes(states, 1, 1, f32, resident.threads) > kResidentSmem) return false;
    resident.cap_cols = 32;
    resident.cap_own = 0;
    bounds.clear();
    bounds.reserve((size_t)n_units * (c + 1));
    for (const Work& w : us) {
      const DevModel* m = models[w.u.p];
      const int32_t* sp = m->h_stateptr.data();
      const int32_t* cp = m->h_colptr.data();
      const uint8_t* fx = fixed_h.data() + base_h[w.u.p];
      auto cost = [&](int32_t s) -> int64_t {
        return fx[s] ? 1 : cp[sp[s + 1]] - cp[sp[s]] + 24 * (sp[s + 1] - sp[s]);
      };
      int64_t total = 0, done = 0;
      if (c > 1)
        for (int32_t s = w.u.s0; s < w.u.s1; ++s) total += cost(s);
      int32_t s = w.u.s0, prev = s;
      bounds.push_back(s);
      for (int r = 1; r <= c; ++r) {
        if (r == c)
          s = w.u.s1;
        else
          while (s < w.u.s1 && done * c < total * r) done += cost(s++);
        bounds.push_back(s);
        resident.cap_own = std::max(resident.cap_own, s - prev);
        resident.cap_cols = std::max(resident.cap_cols, sp[s] - sp[prev]);
        rank_entries = std::max<int64_t>(rank_entries, cp[sp[s]] - cp[sp[prev]]);
        prev = s;
      }
    }
    size_t need = resident_bytes(states, resident.cap_cols, resident.cap_own, f32, resident.threads);
    if (two && !few && need > kResidentHalfSmem) {
      // alone on its SM, a CTA of half the threads leaves half of it idle (1,000 parts
      // of 1,500 states and 5 entries a column: 33.6 ms, 23.2 with all threads)
      resident.threads = kResidentThreads;
      need = resident_bytes(states, resident.cap_cols, resident.cap_own, f32, resident.threads);
    }
    if (need > kResidentSmem || resident.cap_cols > 65535) return false;
    // one unit: its entries go to shared memory as well where they fit (no L2
    // latency in its iterations; pendulum_240 alone 1.03 ms against 1.11). With
    // many units the wider clusters that takes cost more than it saves.
    const size_t all = need + 64 + (size_t)rank_entries * 20;
    copied = n_units == 1 && all <= kResidentSmem;
    resident.smem = (uint32_t)(copied ? all : need);
    // lanes to a column: whole warps when the columns are long or too few for groups
    const double k = (double)entries / std::max<int64_t>(cols, 1);
    resident.group = k >= 256 || (double)cols / n_units / c < 4.0 * resident.threads / 32 / 2 ? 32 : 8;
    resident.cluster = c;
    if (resident_prepare(resident) == cudaSuccess) return true;
    cudaGetLastError();  // wide clusters may not fit the device: the next shape is tried without this error
    return false;
  };
  resident.parts = parts ? 1 : 0;
  resident.f32 = f32 ? 1 : 0;
  resident.cap_states = states;
  resident.max_col = max_col;
  resident.n_units = n_units;
  const auto none = [&]() {
    resident.n_units = 0;
    return IMDP_OK;
  };
  while (!shape(c))
    if ((c *= 2) > kMaxCluster) return none();
  // A unit has its cluster's SMs only, and where there are a few units more than
  // clusters (of 16 CTAs 7 fit the GPU, of 8 15) some wait for another one. A cluster
  // takes 1.25 to 1.46 transitions a cycle and SM. 200 iterations: 5 million
  // transitions with small units beside them 26.8 ms, on the grid kernel 5.2, per
  // iteration 10.4. Beside 40 units of 80,000 and 20 iterations: 1 million, 500
  // iterations 12.8, per iteration 8.4; 300,000, 200 iterations 3.0 and 3.7.
  const auto uneven = [&](int c) {
    const size_t m = resident.clusters;
    const auto seconds = [&](size_t i, double rate) {
      const double its = (double)(us[i].work / std::max<int64_t>(us[i].entries, 1));
      return its * 3e-6 + us[i].work / (rate * c * hz);
    };
    // two CTAs of an SM share its rate while there are units for both
    const double shared = resident.clusters * c > grid ? 1.35 / 2 : 1.35;
    double rest = 0.0;
    for (size_t i = 1; i < us.size(); ++i) rest += seconds(i, shared) / m;
    double first = seconds(0, shared);
    if (first > rest) first = rest + (1.0 - rest / first) * seconds(0, 1.35);
    return c > 1 && us.size() > m ? std::max(first, seconds(m - 1, shared) + seconds(m, shared)) : first;
  };
  // a few units too many for the clusters: more, smaller clusters where that is faster
  // (8 units of 80,000 transitions: 2.05 ms with 7 clusters of 16, 1.40 with 8 of 8;
  // 64 of 6,000: 1.07 with 36 of 4, 0.62 with 64 of 2)
  while (c > 1 && n_units > resident.clusters && n_units <= 2 * resident.clusters &&
         unit_bytes * (2 * grid / c) <= 200e6) {
    const ResidentPlan wide = resident;
    const std::vector<int32_t> wide_bounds = bounds;
    const double before = std::max(uneven(c), spread(c));
    if (shape(c / 2) && std::max(uneven(c / 2), spread(c / 2)) < before) {
      c /= 2;
      continue;
    }
    resident = wide;
    bounds = wide_bounds;
    break;
  }
  // A large problem's first iterations settle most columns, on 16 SMs here: few
  // iterations are left to the grid kernel (1,501 columns of 80 entries, per iteration /
  // resident / grid: 8 iterations 215 / 256 / 128 us, 16 434 / 488 / 244).
  if (alone && !copied && !any_infinite && max_horizon < 24) return none();
  const double mine = std::max(uneven(c), spread(c));
  if (mine > other) return none();
  // (at first all units run, with short horizons beside a long one much more than on average)
  const double all = 3e-6 + (double)entries / (1.17 * std::min<double>(grid, (double)n_units * c) * hz);
  long_seconds = std::max(mine / iters, 0.5 * all);
  std::vector<ResidentUnit> uh(n_units);
  for (int32_t i = 0; i < n_units; ++i) uh[i] = us[i].u;
  ResidentUnit* du = alloc<ResidentUnit>(uh.size());
  int32_t* db = alloc<int32_t>(bounds.size());
  if (!du || !db) {  // no room for the plan: the per-iteration kernels need none
    mem.release(du);
    mem.release(db);
    return none();
  }
  cudaError_t err = cudaMemcpyAsync(du, uh.data(), sizeof(ResidentUnit) * uh.size(), cudaMemcpyHostToDevice, st);
  if (err == cudaSuccess) err = cudaMemcpyAsync(db, bounds.data(), sizeof(int32_t) * bounds.size(), cudaMemcpyHostToDevice, st);
  if (err == cudaSuccess) err = cudaStreamSynchronize(st);  // the host vectors go out of scope
  if (err != cudaSuccess) return cuda_status(err, "session plan");
  resident.units = du;
  resident.bounds = db;
  return IMDP_OK;
}

imdp_status Session::plan_grid(cudaStream_t st) {
  whole = GridPlan{};
  const DevModel* m = models[0];
  GridCut cut;
  const bool f32 = m->lg32 != nullptr;
  if (resident.n_units > 0 || !grid_possible()) return IMDP_OK;
  if (!plan_grid_unit(m, fixed_h.data(), grid, cut)) return IMDP_OK;
  const size_t need = grid_bytes(cut, f32), all = need + 64 + 20 * (size_t)cut.entries;
  copied = all <= kResidentSmem;
  whole.smem = (uint32_t)((copied ? all : need) + 15) & ~15u;
  whole.grid = whole.steal_ctas = grid;
  whole.group = m->nnz >= 256 * (int64_t)m->n_cols || m->n_cols < 48 * (int64_t)grid ? 32 : 8;
  whole.f32 = f32 ? 1 : 0;
  if (grid_prepare(whole) != cudaSuccess) {
    cudaGetLastError();
    return IMDP_OK;
  }
  int32_t* dc = alloc<int32_t>(cut.chunk.size());
  GridWindow* dw = alloc<GridWindow>(cut.win.size());
  GridUnit* du = alloc<GridUnit>(1);
  int2* work = alloc<int2>(grid);
  GridUnit u{};
  u.misses = alloc<GridMiss>((size_t)grid * cut.most_cols);
  u.steal = whole.steal = alloc<uint32_t>(4 * (size_t)grid);
  if (!dc || !dw || !du || !work || !u.misses || !u.steal) {  // as above
    for (void* p : {(void*)dc, (void*)dw, (void*)du, (void*)work, (void*)u.misses, (void*)u.steal}) mem.release(p);
    whole = GridPlan{};
    return IMDP_OK;
  }
  u.chunk = dc;
  u.win = dw;
  u.ctl = ctl;
  u.n_chunks = (int32_t)cut.win.size();
  u.one_window = cut.one_window;
  u.ctas = grid;
  u.single = m->n_cols == m->n_states ? 1 : 0;
  u.most_cols = cut.most_cols;
  u.most_own = cut.most_own;
  u.most_cells = cut.most_cells;
  u.max_col = m->max_col;
  const std::vector<int2> all_of_one(grid, make_int2(0, 1));
  cudaError_t e = cudaMemcpyAsync(dc, cut.chunk.data(), sizeof(int32_t) * cut.chunk.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(dw, cut.win.data(), sizeof(GridWindow) * cut.win.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(du, &u, sizeof(u), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(work, all_of_one.data(), sizeof(int2) * grid, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // the host vectors go out of scope
  if (e != cudaSuccess) return cuda_status(e, "session plan");
  long_seconds = 6.5e-6 + m->nnz / (1.0 * grid * 1.9e9);
  whole.units = du;
  whole.work = work;
  whole.n_units = 1;
  return IMDP_OK;
}

imdp_status Session::install_plan(const std::vector<Tile>& tl, const std::vector<int2>& wl, cudaStream_t st,
                                  bool slice) {
  cudaError_t e = cudaStreamSynchronize(st);  // launches in flight may still read the old plan
  if (e != cudaSuccess) return cuda_status(e, "session plan");
  plan_lost = true;  // until the new one is complete: a step must not read the old one's memory
  mem.drop(items_mem);
  mem.drop(item_end_mem);
  mem.drop(win_mem);
  items = nullptr;
  tile_item_end = nullptr;
  win_cnt = nullptr;
  tiles = (Tile*)mem.refit(tiles_mem, sizeof(Tile) * tl.size());
  wide = (int2*)mem.refit(wide_mem, sizeof(int2) * wl.size());
  if (!tiles || !wide) { set_error("device allocation failed (tile plan)"); return IMDP_ENOMEM; }
  // slice kernel: one work item per slice of every window (tile), in tile order
  std::vector<int2> it;
  std::vector<int32_t> tend;
  if (slice) {
    tend.resize(tl.size());
    for (size_t t = 0; t < tl.size(); ++t) {
      for (int32_t g = tl[t].x0; g < tl[t].x1; ++g) it.push_back(make_int2((int32_t)t, g));
      tend[t] = (int32_t)it.size();
    }
    items = (int2*)mem.refit(items_mem, sizeof(int2) * it.size());
    tile_item_end = (int32_t*)mem.refit(item_end_mem, sizeof(int32_t) * tend.size());
    win_cnt = (unsigned int*)mem.refit(win_mem, sizeof(unsigned int) * tl.size());
    if (!items || !tile_item_end || !win_cnt) { set_error("device allocation failed (slice plan)"); return IMDP_ENOMEM; }
    if (!it.empty()) e = cudaMemcpyAsync(items, it.data(), sizeof(int2) * it.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && !tend.empty())
      e = cudaMemcpyAsync(tile_item_end, tend.data(), sizeof(int32_t) * tend.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(win_cnt, 0, sizeof(unsigned int) * std::max<size_t>(tl.size(), 1), st);
    if (e != cudaSuccess) return cuda_status(e, "session plan");
  }
  L.items = items;
  L.tile_item_end = tile_item_end;
  L.win_cnt = win_cnt;
  L.n_items = (int32_t)it.size();
  if (!tl.empty()) e = cudaMemcpyAsync(tiles, tl.data(), sizeof(Tile) * tl.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && !wl.empty())
    e = cudaMemcpyAsync(wide, wl.data(), sizeof(int2) * wl.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);  // the host vectors belong to the caller
  if (e != cudaSuccess) return cuda_status(e, "session plan");
  // tiles of ranks 0..r (the plan lists problems in rank order)
  std::vector<int32_t> rank(count), end(count, 0);
  for (int r = 0; r < count; ++r) rank[order[r]] = r;
  for (const Tile& T : tl) ++end[rank[T.p]];
  for (int r = 1; r < count; ++r) end[r] += end[r - 1];
  e = cudaMemcpyAsync(rank_of, rank.data(), sizeof(int32_t) * count, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(rank_tile_end, end.data(), sizeof(int32_t) * count, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(&ctl->tile_limit, 0, sizeof(int32_t), st);  // every tile, until a launch ends
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_status(e, "session plan");
  L.rank_of = rank_of;
  L.rank_tile_end = rank_tile_end;
  n_tiles = (int32_t)tl.size();
  n_wide = (int32_t)wl.size();
  wide_entries = 0;
  for (const int2& w : wl) {
    const DevModel* m = models[w.x];
    wide_entries += m->h_colptr[m->h_stateptr[w.y + 1]] - m->h_colptr[m->h_stateptr[w.y]];
  }
  L.tiles = tiles;
  L.n_tiles = n_tiles;
  L.wide = wide;
  L.n_wide = n_wide;
  L.tile_cols = 0;
  for (const Tile& T : tl) L.tile_cols += T.c1 - T.c0;
  if (n_wide > 0 && n_tiles > 0 && !side.stream && (e = side.create()) != cudaSuccess)
    return cuda_status(e, "session side stream");
  if (graph) {
    cudaGraphExecDestroy(graph);
    graph = nullptr;
  }
  plan_lost = false;
  return IMDP_OK;
}

imdp_status Session::prepare_slices(cudaStream_t st) {
  if (qbuf) return IMDP_OK;
  for (int p = 0; p < count; ++p) {
    const SliceLayout* l = nullptr;
    imdp_status r = model_slice_layout(models[p], st, &l);
    if (r != IMDP_OK) return r;
  }
  uint64_t* q = alloc<uint64_t>((size_t)total_cols);
  if (!q) { set_error("device allocation failed (slice kernel)"); return IMDP_ENOMEM; }
  cudaError_t e = cudaStreamSynchronize(st);  // launches in flight read the problem descriptors
  if (e != cudaSuccess) return cuda_status(e, "slice kernel setup");
  int64_t col_off = 0;
  for (int p = 0; p < count; ++p) {
    const SliceLayout* l = models[p]->slices;
    Problem& P = probs_h[p];
    P.sl_slot = l->slot;
    P.sl_meta = l->meta;
    P.sl_rows = l->rows;
    P.sl_lg = l->lg;
    P.qcol = q + col_off;  // same offsets as the hints
    col_off += (int64_t)padded_i32(models[p]->n_cols);
  }
  e = cudaMemcpyAsync(probs, probs_h.data(), sizeof(Problem) * count, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_status(e, "slice kernel setup");
  qbuf = q;
  return IMDP_OK;
}

void Session::build_plan(const LaunchConfig& c, std::vector<Tile>& tl, std::vector<int2>& wl) const {
  const LaunchConfig r = resolve_launch(L, &c);
  if (r.kernel == kKernelSlice) {
    // the windows of every problem's slice layout (prepare_slices built them);
    // x0 / x1 are the window's slices
    for (int p : order) {
      const DevModel* m = models[p];
      const SliceLayout* l = m->slices;
      for (int32_t w = 0; w < l->n_windows; ++w) {
        Tile T;
        T.p = p;
        T.s0 = l->h_win_s0[w];
        T.s1 = l->h_win_s0[w + 1];
        T.c0 = m->h_stateptr[T.s0];
        T.c1 = m->h_stateptr[T.s1];
        T.e0 = m->h_colptr[T.c0];
        T.e1 = m->h_colptr[T.c1];
        T.x0 = l->h_win_sl0[w];
        T.x1 = l->h_win_sl0[w + 1];
        tl.push_back(T);
      }
    }
    return;
  }
  for (int p : order) {
    std::vector<int32_t> ws;
    const size_t at = tl.size();
    plan_tiles(models[p], p, tl, ws, r.tile_entries, r.wide_col, fixed_h.data() + base_h[p]);
    for (size_t t = at; t < tl.size(); ++t) tl[t].p = p;
    for (int32_t s : ws) wl.push_back(make_int2(p, s));
  }
}

imdp_status Session::set_launch(const LaunchConfig& c, cudaStream_t st) {
  const LaunchConfig old = resolve_launch(L, &cfg), now = resolve_launch(L, &c);
  const bool slice = now.kernel == kKernelSlice;
  if (plan_lost || now.tile_entries != old.tile_entries || now.wide_col != old.wide_col || slice != (old.kernel == kKernelSlice)) {
    if (slice) {
      imdp_status r = prepare_slices(st);
      if (r != IMDP_OK) return r;
    }
    std::vector<Tile> tl;
    std::vector<int2> wl;
    build_plan(c, tl, wl);
    imdp_status r = install_plan(tl, wl, st, slice);
    if (r != IMDP_OK) return r;
  }
  cfg = c;
  if (graph) {
    cudaGraphExecDestroy(graph);
    graph = nullptr;
  }
  return IMDP_OK;
}

imdp_status Session::reset(cudaStream_t st) {
  TraceRange trace("imdp session reset");
  // the failure-detection test hook ends with a reset; a graph captured while it
  // was on replays launches that issue no copies, so it is captured again
  g_stall_producer.store(0);
  if (graph && graph_stalled) {
    cudaGraphExecDestroy(graph);
    graph = nullptr;
  }
  // both buffers: states the property fixes are in no tile, so no launch writes them
  init_values_kernel<<<(int)std::min<int64_t>((total + 255) / 256, 8192), 256, 0, st>>>(total, fixed, V);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) {
    init_values_kernel<<<(int)std::min<int64_t>((total + 255) / 256, 8192), 256, 0, st>>>(total, fixed, V + total);
    e = cudaGetLastError();
  }
  for (int p = 0; p < count && e == cudaSuccess; ++p)
    if (w0[p]) e = cudaMemcpyAsync(probs_h[p].V[0], w0[p], sizeof(uint64_t) * probs_h[p].n_states,
                                   cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(hints, 0xff, sizeof(int32_t) * (size_t)total_cols, st);  // -1: no hint
  if (e == cudaSuccess) e = cudaMemsetAsync(its, 0, sizeof(IterState) * count, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(ctl, 0, sizeof(StepControl), st);
  for (int p = 0; p < count && e == cudaSuccess; ++p)
    if (policy_cells[p] > 0) {
      fill_i32_kernel<<<(int)std::min<int64_t>((policy_cells[p] + 255) / 256, 4096), 256, 0, st>>>(
          policy_cells[p], probs_h[p].policy, -1);
      e = cudaGetLastError();
    }
  if (e != cudaSuccess) return cuda_status(e, "session reset");
  launched_since_reset = 0;
  return IMDP_OK;
}

int32_t Session::step_kernel(int32_t n) const {
  if ((cfg.by_rule() || cfg.long_by_rule) && n >= kResidentSteps) {
    if (resident.n_units > 0) return kKernelResident;
    if (whole.n_units > 0) return kKernelGrid;
  }
  return resolve_launch(L, &cfg).kernel;
}

// Iterations of one launch of a long step call. Another stream's grid kernel waits
// for all SMs together, so a launch takes about 10 ms, which costs nothing that can
// be measured (cartpole_3840 11.48 ms in one launch and 11.49 so). A launch whose
// units follow one another on the clusters reads their transitions from memory
// again and has a last round of its own: about 100 ms (4096 pendulum parts, 65.3 ms
// in one launch: 67.0 in launches of 30 ms, 69.0 of 10; on 32-bit storage 65.8,
// 70.9, 74.2; 256 uneven problems 71.4, 74.2, 76.8), and 100 times as long as that
// reading takes (10,000 uneven problems, 32 GB: 2.30 s in launches of half a second,
// 2.39 of a tenth).
int32_t Session::launch_iterations() const {
  double most = 0.01;
  if (resident.n_units > resident.clusters) {
    double bytes = 0.0;
    for (const DevModel* m : models) bytes += m->nnz * (m->lg32 ? 12.0 : 20.0);
    most = std::max(0.1, 100.0 * bytes / 6.8e12);
  }
  return (int32_t)std::min(50000.0, std::max(16.0, most / std::max(long_seconds, 1e-9)));
}

imdp_status Session::step(int32_t n, cudaStream_t st) {
  if (n <= 0) return IMDP_OK;
  TraceRange trace("imdp session step");
  cudaError_t e = cudaSuccess;
  const int32_t kernel = step_kernel(n);
  int32_t done = 0;
  if (kernel == kKernelTiny) {
    // one small problem, few iterations: all of them in one launch of one CTA
    e = launch_bellman_tiny(L, n, models[0]->lg32 != nullptr, st);
    if (e != cudaSuccess) return cuda_status(e, "bellman step");
    launches += n;
    launched_since_reset += n;
    return IMDP_OK;
  }
  if (kernel == kKernelResident || kernel == kKernelGrid) {
    // by rule: all n iterations in one launch, or in a few
    const int32_t most = launch_iterations();
    while (done < n && e == cudaSuccess) {
      const int32_t some = std::min(most, n - done);
      e = kernel == kKernelResident ? launch_bellman_resident(L, resident, some, st)
                                    : launch_bellman_grid(L, whole, some, st);
      if (e == cudaSuccess) done += some;
    }
    if (e == cudaErrorCooperativeLaunchTooLarge) {  // nothing was launched: per iteration from here on
      cudaGetLastError();
      whole.n_units = 0;
      e = cudaSuccess;
    }
  }
  if (done < n && plan_lost) {
    set_error("the session has no launch plan (a change of its configuration found no memory); set one");
    return IMDP_ENOMEM;
  }
  if (e == cudaSuccess && st != nullptr && n - done >= kGraphChunk) {
    if (!graph) {
      cudaGraph_t g = nullptr;
      graph_stalled = g_stall_producer.load() != 0;
      e = cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal);
      for (int i = 0; i < kGraphChunk && e == cudaSuccess; ++i) e = launch_bellman_step(L, grid, st, &side, &cfg);
      cudaError_t e2 = cudaStreamEndCapture(st, &g);
      if (e == cudaSuccess) e = e2;
      if (e == cudaSuccess) e = cudaGraphInstantiate(&graph, g, 0);
      if (g) cudaGraphDestroy(g);
      if (e != cudaSuccess) {
        graph = nullptr;
        return cuda_status(e, "graph capture");
      }
    }
    for (; done + kGraphChunk <= n && e == cudaSuccess; done += kGraphChunk) e = cudaGraphLaunch(graph, st);
  }
  for (; done < n && e == cudaSuccess; ++done) e = launch_bellman_step(L, grid, st, &side, &cfg);
  if (e != cudaSuccess) return cuda_status(e, "bellman step");
  launches += n;
  launched_since_reset += n;
  return IMDP_OK;
}

imdp_status Session::read_states(std::vector<IterState>& out, cudaStream_t st) {
  out.resize(count);
  StepControl c{};
  cudaError_t e = cudaMemcpyAsync(out.data(), its, sizeof(IterState) * count, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&c, ctl, sizeof(StepControl), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_status(e, "read iteration state");
  if (c.error) {
    set_error("a bounded wait inside the Bellman kernel gave up (results of this session are invalid)");
    return IMDP_ETIMEOUT;
  }
  return IMDP_OK;
}

imdp_status Session::run(int32_t check_every, cudaStream_t st) {
  for (const Problem& P : probs_h)
    if (P.external_stop) {
      set_error("an infinite horizon on a state-sharded slice stops on the residual of every slice: step it and "
                "test imdp_session_residual across the slices");
      return IMDP_EINVAL;
    }
  if (!any_infinite) {
    // Every problem finishes within max_horizon launches of the reset.
    return step(std::max<int32_t>(0, max_horizon - (int32_t)std::min<int64_t>(launched_since_reset, max_horizon)), st);
  }
  if (check_every <= 0) check_every = 32;
  std::vector<IterState> s;
  while (launched_since_reset < max_horizon) {
    const int32_t n = (int32_t)std::min<int64_t>(check_every, max_horizon - launched_since_reset);
    imdp_status r = step(n, st);
    if (r != IMDP_OK) return r;
    r = read_states(s, st);
    if (r != IMDP_OK) return r;
    bool all = true;
    for (int p = 0; p < count; ++p) all = all && s[p].done;
    if (all) break;
  }
  return IMDP_OK;
}

imdp_status Session::read(int32_t p, double* V_out, int32_t* k_out, double* res_out, int32_t* pol_out,
                          cudaStream_t st) {
  if (p < 0 || p >= count) { set_error("problem index out of range"); return IMDP_EINVAL; }
  std::vector<IterState> s;
  imdp_status r = read_states(s, st);
  if (r != IMDP_OK) return r;
  const Problem& P = probs_h[p];
  const int32_t k = s[p].done ? s[p].k_final : s[p].iter;
  if (k_out) *k_out = k;
  const int32_t n = P.n_states;
  const uint64_t* Vk = P.V[k & 1];
  const uint64_t* Vk1 = P.V[(k + 1) & 1];
  const int g = std::min((n + 255) / 256, 4096);
  std::vector<void*> tmp;
  auto cleanup = [&]() { for (void* t : tmp) cudaFree(t); };
  auto emit = [&](double* out, const uint64_t* prev) -> cudaError_t {
    if (!out) return cudaSuccess;
    double* dst = out;
    const bool host = !is_device_pointer(out);
    if (host) {
      void* t = nullptr;
      cudaError_t ea = cudaMalloc(&t, sizeof(double) * std::max(n, 1));
      if (ea != cudaSuccess) return ea;
      tmp.push_back(t);
      dst = (double*)t;
    }
    if (prev == nullptr || k >= 1) {
      export_values_kernel<<<g, 256, 0, st>>>(n, Vk, prev, v_offset[p], v_scale[p], dst);
    } else {
      cudaMemsetAsync(dst, 0, sizeof(double) * n, st);
    }
    cudaError_t e2 = cudaGetLastError();
    if (e2 == cudaSuccess && host) e2 = cudaMemcpyAsync(out, dst, sizeof(double) * n, cudaMemcpyDeviceToHost, st);
    return e2;
  };
  cudaError_t e = emit(V_out, nullptr);
  if (e == cudaSuccess) e = emit(res_out, Vk1);
  if (e == cudaSuccess && pol_out) {
    if (!P.policy) {
      cleanup();
      set_error("policy was not requested when the session was created");
      return IMDP_EINVAL;
    }
    e = cudaMemcpyAsync(pol_out, P.policy, sizeof(int32_t) * policy_cells[p], cudaMemcpyDefault, st);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cleanup();
  if (e != cudaSuccess) return cuda_status(e, "session read");
  if (s[p].noconv) {
    set_error("infinite horizon did not converge within the iteration cap");
    return IMDP_ENOCONV;
  }
  return IMDP_OK;
}

imdp_status Session::read_all(double* const* V_out, int32_t* k_out, cudaStream_t st) {
  std::vector<IterState> s;
  imdp_status r = read_states(s, st);
  if (r != IMDP_OK) return r;
  // host outputs pass through one device buffer and one host buffer
  std::vector<int64_t> staged(count, -1);
  std::vector<std::pair<uintptr_t, uintptr_t>> spans;
  int64_t host = 0;
  int32_t most = 1;
  for (int p = 0; p < count; ++p) {
    const int32_t n = probs_h[p].n_states;
    most = std::max(most, n);
    spans.emplace_back((uintptr_t)V_out[p], (uintptr_t)(V_out[p] + n));
    if (!is_device_pointer(V_out[p])) {
      staged[p] = host;
      host += n;
    }
  }
  std::sort(spans.begin(), spans.end());
  bool apart = count <= 65535;  // (the launch's limit)
  for (int p = 1; p < count; ++p) apart = apart && spans[p].first >= spans[p - 1].second;
  ExportItem* d_items = nullptr;
  double* stage = nullptr;
  cudaError_t e = cudaSuccess;
  if (apart) {
    e = cudaMalloc(&d_items, sizeof(ExportItem) * count);
    if (e == cudaSuccess && host > 0) e = cudaMalloc(&stage, sizeof(double) * host);
    apart = e == cudaSuccess;
  }
  // outputs that overlap are written one problem after the other, and so are
  // those that find no room together
  if (!apart) {
    cudaGetLastError();
    cudaFree(d_items);
    imdp_status worst = IMDP_OK;
    for (int p = 0; p < count; ++p) {
      int32_t k = 0;
      r = read(p, V_out[p], &k, nullptr, nullptr, st);
      if (r != IMDP_OK && r != IMDP_ENOCONV) return r;
      if (r != IMDP_OK) worst = r;
      if (k_out) k_out[p] = k;
    }
    return worst;
  }
  std::vector<ExportItem> items(count);
  for (int p = 0; p < count; ++p) {
    const Problem& P = probs_h[p];
    const int32_t k = s[p].done ? s[p].k_final : s[p].iter;
    items[p] = ExportItem{P.V[k & 1], staged[p] >= 0 ? stage + staged[p] : V_out[p], v_offset[p], v_scale[p], P.n_states};
  }
  std::vector<double> back((size_t)host);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(d_items, items.data(), sizeof(ExportItem) * count, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) {
    export_batch_kernel<<<dim3((unsigned)std::min((most + 255) / 256, 64), (unsigned)count), 256, 0, st>>>(d_items);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && host > 0)
    e = cudaMemcpyAsync(back.data(), stage, sizeof(double) * host, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(d_items);
  cudaFree(stage);
  if (e != cudaSuccess) return cuda_status(e, "session read");
  imdp_status worst = IMDP_OK;
  for (int p = 0; p < count; ++p) {
    if (staged[p] >= 0) std::memcpy(V_out[p], back.data() + staged[p], sizeof(double) * probs_h[p].n_states);
    if (k_out) k_out[p] = s[p].done ? s[p].k_final : s[p].iter;
    if (s[p].noconv) worst = IMDP_ENOCONV;
  }
  if (worst == IMDP_ENOCONV) set_error("infinite horizon did not converge within the iteration cap");
  return worst;
}

}  // namespace imdp
