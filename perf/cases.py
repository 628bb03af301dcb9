"""The work that users of this framework have it do, as timed cases.

Every case goes through the package's public entry points: one query on a resident
model, a resident session stepped again and again, a batch of independent problems,
a burst of requests to the server, and a model that is created and queried once.
Model shapes are those of the paper's benchmark table (linear_5, pendulum_240,
cartpole_960 and _3840, harrier, pimdp_2), the uneven batch and the served stream of
the benchmark, and a sparse unstructured model; ``draw`` takes others of the same
ranges.  Launch configurations are left to the library's rule.

Inputs are generated on the GPU from the seed alone: banded models (a Gaussian
window of destinations around the source state plus an absorbing sink, as
``workloads.imdp_synth`` draws them) and models with scattered destinations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2401_04068_gb300 as g

PROPERTY = {"reach": g.IMDP_REACH, "avoid": g.IMDP_REACH_AVOID, "reward": g.IMDP_REWARD}

# One case: `path` is the entry point; `model` the structure (banded, scattered, or
# uneven: one banded shape per problem); `blocks` the number of models; `merged`:
# they form one block-diagonal model; `states` grid states per block, `actions` per
# state, `window` the mean in-domain destinations of a column (lengths vary by half
# of it either way), `eps` the relative width of the intervals, `shapes` the seed of an
# uneven set's shapes and horizons (the sizes of a case are its own, its values the seed's).
DEFAULTS = dict(path="session", model="banded", blocks=1, merged=False, states=240, actions=1, window=109.0, eps=0.05,
                storage="f64", horizon=200, infinite=False, tol=1e-6, property="reach", discount=0.95,
                pessimistic=True, maximize=True, policy=False, shapes=0)


def _case(name=None, **kw):
    c = dict(DEFAULTS)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest model of the table, asked once: latency of one call
        _case("query_linear5", path="query", states=5, window=5.0, eps=0.1, policy=True),
        # one pendulum abstraction, control synthesis with the time-dependent policy
        _case("query_pendulum240", path="query", states=240, window=108.7, policy=True),
        # a model from host arrays, created and queried once (what a command line run does)
        _case("create_cartpole960", path="create", states=960, window=560.0, eps=0.1),
        # expected discounted reward, worst strategy under an optimistic adversary, on a sparse unstructured model
        _case("reward_scattered", model="scattered", states=20000, actions=2, window=12.0, eps=0.3, horizon=100,
              property="reward", pessimistic=False, maximize=False, policy=True),
        # many independent problems of different shapes and horizons in one call
        _case("batch_uneven", path="batch", model="uneven", blocks=256, states=960, actions=4, window=400.0,
              horizon=500, shapes=7),
        # 4096 pendulum abstractions as one block-diagonal model: throughput, both storages
        _case("blocks_pendulum240", blocks=4096, merged=True, states=240, window=108.7),
        _case("blocks_pendulum240_f32", blocks=4096, merged=True, states=240, window=108.7, storage="f32"),
        # the largest model of the table, both storages
        _case("pimdp2", states=42633, actions=3, window=375.1),
        _case("pimdp2_f32", states=42633, actions=3, window=375.1, storage="f32"),
        # reach-avoid to convergence, with the stationary policy
        _case("harrier_infinite", states=25920, window=715.6, infinite=True, horizon=300, property="avoid", policy=True),
        # long columns, optimistic bound
        _case("cartpole3840_optimistic", states=3840, window=2242.5, eps=0.1, pessimistic=False),
        # a burst of requests of mixed sizes to the continuous-batching server
        _case("served_burst", path="served", model="uneven", blocks=64, states=4000, actions=3, window=700.0,
              horizon=500, shapes=8),
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["tiny", "query", "create", "reward", "batch", "blocks", "blocks", "single", "single", "long",
                       "served"])
    modes = dict(pessimistic=rng.random() < 0.6, maximize=rng.random() < 0.7, eps=rng.choice([0.05, 0.1]))
    storage = rng.choice(["f64", "f64", "f32"])
    K = rng.randint(50, 200)
    if kind == "tiny":
        n = rng.randint(3, 60)
        return _case(path="query", states=n, actions=rng.randint(1, 3), window=rng.uniform(1.5, min(n, 12)), horizon=K,
                     policy=rng.random() < 0.5, storage=storage, **modes)
    if kind == "query":
        n = int(_logu(rng, 80, 3000))
        return _case(path="query", states=n, actions=rng.randint(1, 3), window=_logu(rng, 4, min(n, 400)), horizon=K,
                     policy=rng.random() < 0.5, storage=storage, property=rng.choice(["reach", "avoid"]), **modes)
    if kind == "create":
        n = int(_logu(rng, 100, 2500))
        return _case(path="create", states=n, actions=rng.randint(1, 2), window=_logu(rng, 5, 0.5 * n), horizon=K,
                     storage=storage, **modes)
    if kind == "reward":
        return _case(model="scattered", states=int(_logu(rng, 1000, 50000)), actions=rng.randint(1, 4),
                     window=_logu(rng, 4, 40), horizon=K, property="reward", discount=rng.uniform(0.8, 0.99),
                     policy=rng.random() < 0.5, storage=storage, pessimistic=modes["pessimistic"],
                     maximize=modes["maximize"], eps=0.3)
    if kind == "batch":
        return _case(path="batch", model="uneven", blocks=int(_logu(rng, 16, 256)), states=960, actions=4,
                     window=400.0, horizon=rng.randint(100, 500), storage=storage, shapes=rng.randrange(1 << 30), **modes)
    if kind == "blocks":
        n = rng.randint(60, 500)
        w = _logu(rng, 8, 0.6 * n)
        return _case(blocks=max(16, int(_logu(rng, 2e6, 1e8) / (n * w))), merged=True, states=n, window=w, horizon=K,
                     storage=storage, **modes)
    if kind == "single":
        n, a, w = int(_logu(rng, 4000, 42000)), rng.randint(1, 3), _logu(rng, 30, 720)
        w = min(w, 4.5e7 / (n * a))
        return _case(states=n, actions=a, window=w, horizon=K, storage=storage,
                     property=rng.choice(["reach", "avoid"]), infinite=rng.random() < 0.25, **modes)
    if kind == "long":
        n = rng.randint(1500, 3800)
        return _case(states=n, actions=rng.randint(1, 2), window=n * rng.uniform(0.35, 0.65), horizon=K,
                     storage=storage, **modes)
    return _case(path="served", model="uneven", blocks=int(_logu(rng, 8, 64)), states=4000, actions=3, window=700.0,
                 horizon=500, shapes=rng.randrange(1 << 30), **modes)


def _shapes(case):
    """Per block: grid states, actions, mean window, eps, horizon (host arrays)."""
    B = case["blocks"]
    if case["model"] != "uneven":
        one = np.ones(B, np.int64)
        return (case["states"] * one, case["actions"] * one, case["window"] * one.astype(float),
                np.full(B, case["eps"]), case["horizon"] * one)
    rng = np.random.default_rng(case["shapes"])
    if case["path"] == "served":  # log-uniform sizes
        nd = np.exp(rng.uniform(np.log(50), np.log(case["states"]), B)).astype(np.int64)
        kb = np.minimum(np.exp(rng.uniform(np.log(3), np.log(case["window"]), B)), nd)
    else:
        nd = rng.integers(5, case["states"] + 1, B)
        kb = rng.uniform(2, np.minimum(case["window"], nd), B)
    na = rng.integers(1, case["actions"] + 1, B)
    return nd, na, kb, rng.choice([0.05, 0.1], B), rng.integers(max(1, case["horizon"] // 5), case["horizon"] + 1, B)


def _repeat(x, counts):
    return torch.repeat_interleave(x, counts)


def _generate(case, seed):
    """The case's models as one block-diagonal CSC model on the GPU, and its queries."""
    dev = "cuda"
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))

    def u(n):
        return torch.rand(n, generator=gen, device=dev, dtype=torch.float64)

    nd_h, na_h, kb_h, eps_h, hor_h = _shapes(case)
    nd, na = (torch.as_tensor(x, device=dev, dtype=torch.int64) for x in (nd_h, na_h))
    kb, eps = (torch.as_tensor(x, device=dev, dtype=torch.float64) for x in (kb_h, eps_h))
    banded = case["model"] != "scattered"
    B = len(nd_h)
    ns = nd + 1 if banded else nd              # states per block (banded: plus the sink)
    ncol = nd * na + (1 if banded else 0)
    block = _repeat(torch.arange(B, device=dev), ncol)
    cbase = torch.cumsum(ncol, 0) - ncol
    local = torch.arange(block.numel(), device=dev) - cbase[block]
    nd_c, na_c = nd[block], na[block]
    kk = torch.clamp(torch.round(kb[block] * (0.5 + u(block.numel()))).long(), min=1)
    kk = torch.minimum(kk, nd_c)
    sink_col = local == nd_c * na_c
    cnt = torch.where(sink_col, 1, kk + 1) if banded else kk
    colptr = torch.zeros(block.numel() + 1, dtype=torch.int64, device=dev)
    torch.cumsum(cnt, 0, out=colptr[1:])
    col = _repeat(torch.arange(block.numel(), device=dev), cnt)
    pos = torch.arange(col.numel(), device=dev) - colptr[col]
    sbase = torch.cumsum(ns, 0) - ns
    if banded:
        sigma = torch.clamp(kk / 4.0, min=0.5)
        action = local % na_c
        centre = (local // na_c).double() + (action - (na_c - 1) / 2.0) * torch.clamp(kk / 3.0, min=1.0)
        centre += 0.25 * sigma * (2.0 * u(block.numel()) - 1.0)
        start = torch.minimum(torch.clamp(torch.round(centre - kk / 2.0).long(), min=0), nd_c - kk)
        to_sink = (pos == kk[col]) | sink_col[col]
        dest = torch.where(to_sink, nd_c[col], start[col] + pos)
        w = torch.exp(-0.5 * ((dest - centre[col]) / sigma[col]) ** 2).masked_fill_(to_sink, 0.0)
        wsum = torch.segment_reduce(w, "sum", lengths=cnt)
        dist = torch.clamp(torch.minimum(centre, (nd_c - 1) - centre), min=0.0)
        leak = torch.where(sink_col, 1.0, 1e-3 + 0.3 * torch.exp(-dist / sigma))
        p = torch.where(to_sink, leak[col], w / wsum[col] * (1.0 - leak[col]))
        del w, wsum
    else:  # one destination in each of a column's equal strips of the state space
        strip = nd_c[col] / kk[col].double()
        dest = torch.floor((pos + u(col.numel()) * (1.0 - 1.0 / strip)) * strip).long()
        w = 0.05 + u(col.numel())
        p = w / torch.segment_reduce(w, "sum", lengths=cnt)[col]
    e = eps[block][col]
    lower = p * (1.0 - e * u(col.numel()))
    upper = torch.clamp(p * (1.0 + e * u(col.numel())), max=1.0)
    if banded:  # the sink column is exact
        fixed = sink_col[col]
        lower[fixed] = 1.0
        upper[fixed] = 1.0
    rowval = (sbase[block][col] + dest).int()
    acts = torch.ones(int(ns.sum()), dtype=torch.int64, device=dev)
    sblock = _repeat(torch.arange(B, device=dev), ns)
    sloc = torch.arange(acts.numel(), device=dev) - sbase[sblock]
    acts = torch.where(sloc < nd[sblock], na[sblock], 1)
    stateptr = torch.zeros(acts.numel() + 1, dtype=torch.int64, device=dev)
    torch.cumsum(acts, 0, out=stateptr[1:])
    goal = torch.clamp(torch.round(0.1 * nd.double()).long(), min=1)
    g0 = ((nd - goal) // 2)[sblock]
    mask = torch.zeros(acts.numel(), dtype=torch.int8, device=dev)
    if case["property"] != "reward":
        mask[(sloc >= g0) & (sloc < g0 + goal[sblock])] = 1
    if case["property"] == "avoid":
        mask[sloc == nd[sblock]] = 2
    reward = u(acts.numel()) if case["property"] == "reward" else None
    return dict(stateptr=stateptr.int(), colptr=colptr.int(), rowval=rowval, lower=lower, upper=upper, mask=mask,
                reward=reward, sbase=sbase.cpu().numpy(), ns=ns.cpu().numpy(), sblock=sblock,
                horizon=np.asarray(hor_h, np.int64))


def _problems(case, m):
    """(first state, states, horizon, pessimistic) of every problem."""
    if case["merged"] or case["blocks"] == 1:
        return [(0, int(m["mask"].numel()), int(m["horizon"][0]), case["pessimistic"])]
    mixed = case["path"] == "served"  # the stream asks for either bound
    return [(int(s), int(n), int(h), case["pessimistic"] if not mixed or i % 4 else not case["pessimistic"])
            for i, (s, n, h) in enumerate(zip(m["sbase"], m["ns"], m["horizon"]))]


def _spec(case, m, mask_h, reward_h, s0, n, horizon, pessimistic):
    part = mask_h[s0:s0 + n]
    return dict(property=PROPERTY[case["property"]], infinite_time=case["infinite"], horizon=horizon, eps=case["tol"],
                pessimistic=pessimistic, maximize=case["maximize"], reach=np.flatnonzero(part == 1).astype(np.int32),
                avoid=np.flatnonzero(part == 2).astype(np.int32),
                reward=None if reward_h is None else reward_h[s0:s0 + n], discount=case["discount"])


class _Host:
    """Host arrays of one model, as a file reader hands them over."""

    def __init__(self, m):
        for k in ("stateptr", "colptr", "rowval", "lower", "upper"):
            setattr(self, k, m[k].cpu().numpy())
        self.n_states = self.stateptr.size - 1


def prepare(case, seed):
    m = _generate(case, seed)
    mask_h = m["mask"].cpu().numpy()
    reward_h = None if m["reward"] is None else m["reward"].cpu().numpy()
    dtype = g.IMDP_F32 if case["storage"] == "f32" else g.IMDP_F64
    probs = _problems(case, m)
    specs = [_spec(case, m, mask_h, reward_h, *p) for p in probs]
    st = dict(case=case, specs=specs, sizes=[p[1] for p in probs], dtype=dtype)
    if case["path"] == "create":
        st["host"] = _Host(m)
        return st
    models = []
    sp, cp = m["stateptr"], m["colptr"]
    if len(probs) > 1:  # each problem's own arrays, with its own indices
        sp_h = sp.cpu().numpy()
        cp_h = cp.cpu().numpy()
        local = m["rowval"] - torch.as_tensor(m["sbase"], device="cuda", dtype=torch.int32)[
            m["sblock"][m["rowval"].long()]]
    for s0, n, _, _ in probs:
        if len(probs) == 1:
            models.append(g.imdp_create_csc(n, cp.numel() - 1, m["rowval"].numel(), sp, cp, m["rowval"], m["lower"],
                                            m["upper"], dtype))
            continue
        c0, c1 = int(sp_h[s0]), int(sp_h[s0 + n])
        e0, e1 = int(cp_h[c0]), int(cp_h[c1])
        models.append(g.imdp_create_csc(n, c1 - c0, e1 - e0, np.ascontiguousarray(sp_h[s0:s0 + n + 1] - c0),
                                        np.ascontiguousarray(cp_h[c0:c1 + 1] - e0), local[e0:e1], m["lower"][e0:e1],
                                        m["upper"][e0:e1], dtype))
    st["models"] = models
    n = sum(st["sizes"])
    if case["path"] != "query":
        st["V"] = torch.zeros(n, dtype=torch.float64, device="cuda")
        st["views"] = list(torch.split(st["V"], st["sizes"]))
        st["k"] = np.zeros(len(probs), np.int32)
        st["made"] = [g.make_spec(**s) for s in specs]
    if case["path"] == "session":
        st["stream"] = torch.cuda.Stream()
        st["residual"] = torch.zeros_like(st["V"])
        if case["policy"]:
            rows = 1 if case["infinite"] else case["horizon"]
            st["policy"] = torch.zeros((rows, n), dtype=torch.int32, device="cuda")
        st["session"] = g.imdp_session_create(models, st["made"], [1] if case["policy"] else None, st["stream"])
    if case["path"] == "served":
        st["server"] = g.imdp_server_create(256 << 20)
    return st


def run(state):
    case = state["case"]
    path = case["path"]
    if path in ("query", "create"):
        model = state["models"][0] if path == "query" else g.create_model(state["host"], state["dtype"])
        _, V, k, residual, policy = g.value_iteration(model, state["sizes"][0], policy=case["policy"],
                                                      **state["specs"][0])
        return dict(V=V, residual=residual, policy=policy, k=k)
    if path == "session":
        s, stream, k = state["session"], state["stream"], [0]
        g.imdp_session_reset(s, stream)
        g.imdp_session_run(s, 0, stream)
        g.imdp_session_read(s, 0, state["V"], k, state["residual"], state.get("policy"), stream)
        return dict(V=state["V"], residual=state["residual"], policy=state.get("policy"), k=k[0])
    if path == "batch":
        g.imdp_value_iteration_batch(state["models"], state["made"], state["views"], state["k"])
        return dict(V=state["V"], k=state["k"])
    server = state["server"]
    tickets = [g.imdp_server_submit(server, m, s) for m, s in zip(state["models"], state["made"])]
    for i, t in enumerate(tickets):
        k = [0]
        status = g.imdp_server_wait(server, t, 60000.0, state["views"][i], k)
        if status != g.IMDP_OK:
            raise RuntimeError("request %d: status %d" % (i, status))
        state["k"][i] = k[0]
    return dict(V=state["V"], k=state["k"])


def _expected(case):
    """(transitions, columns, states, transitions x iterations) of a case: means over the seeds."""
    nd, na, kb, _, hor = (x.astype(float) for x in _shapes(case))
    banded = case["model"] != "scattered"
    nnz = nd * na * (np.minimum(kb, nd) + banded)
    K = 100.0 if case["infinite"] else hor  # iterations
    return [float(x.sum()) for x in (nnz, nd * na, nd + banded, nnz * K)]


def work(case):
    """The model (as the storage keeps it) read once, the outputs written once; a multiply, an
    addition to the value and one to the gap prefix per transition and iteration."""
    nnz, cols, states, updates = _expected(case)
    entry = 20 if case["storage"] == "f64" or case["path"] == "create" else 12
    out = 8 * states * (1 if case["path"] in ("batch", "served") else 2)
    if case["policy"]:
        out += 4 * states * (1 if case["infinite"] else case["horizon"])
    return {"bytes": entry * nnz + 12 * cols + 4 * states + out, "flops": 3 * updates}


class _Columns:
    """Columns of similar length side by side (padded to the longest), for the exact values."""

    def __init__(self, m, cols, lens):
        off = torch.arange(int(lens.max()), device="cuda")
        at = m["colptr"][cols].long()[:, None] + off[None, :]
        ok = off[None, :] < lens[:, None]
        at = torch.where(ok, at, 0)
        self.cols = cols
        self.rows = m["rowval"][at]
        self.lower = torch.where(ok, m["lower"][at], 0.0)
        self.gap = torch.where(ok, m["upper"][at] - m["lower"][at], 0.0)
        self.rem = 1.0 - self.lower.sum(1, keepdim=True)

    def q(self, V, sign, running):
        """O-maximization of the columns in `running`: sort by value, hand out what the lower bounds leave."""
        if not bool(running.any()):
            return None, None
        r, lower, gap, rem, sg = self.rows, self.lower, self.gap, self.rem, sign
        if not bool(running.all()):
            r, lower, gap, rem, sg = r[running], lower[running], gap[running], rem[running], sg[running]
        v = V[r.long()]
        key, order = torch.sort(v * sg, dim=1)
        gs = torch.gather(gap, 1, order)
        give = torch.minimum(torch.clamp(rem - (torch.cumsum(gs, 1) - gs), min=0.0), gs)
        return self.cols[running], (v * lower).sum(1) + (key * sg * give).sum(1)


def exact(case, seed):
    if _expected(case)[3] > 2.5e10:
        return None  # over about 20 seconds
    m = _generate(case, seed)
    probs = _problems(case, m)
    dev = "cuda"
    stateptr = m["stateptr"].long()
    n = stateptr.numel() - 1
    state_of = _repeat(torch.arange(n, device=dev), stateptr[1:] - stateptr[:-1])
    problem = torch.zeros(n, dtype=torch.int64, device=dev)
    for i, (s0, ns, _, _) in enumerate(probs):
        problem[s0:s0 + ns] = i
    sign = torch.tensor([1.0 if p[3] else -1.0 for p in probs], device=dev, dtype=torch.float64)[problem]
    hor = torch.tensor([p[2] for p in probs], device=dev)[problem]
    lens = (m["colptr"][1:] - m["colptr"][:-1]).long()
    width = torch.pow(2.0, torch.ceil(2.0 * torch.log2(lens.double())) / 2.0)  # half octaves
    groups = [_Columns(m, c, lens[c]) for c in (torch.nonzero(width == x).flatten() for x in torch.unique(width))]
    gs = [(c, sign[state_of[c.cols]][:, None], hor[state_of[c.cols]]) for c in groups]
    mask, reward = m["mask"], m["reward"]
    V = reward.clone() if reward is not None else (mask == 1).double()
    K = int(max(p[2] for p in probs))
    worst = -math.inf if case["maximize"] else math.inf
    how = "amax" if case["maximize"] else "amin"
    residual = torch.zeros_like(V)
    for k in range(K):
        best = torch.full((n,), worst, dtype=torch.float64, device=dev)
        for c, sg, h in gs:
            cols, q = c.q(V, sg, h > k)
            if q is not None:
                best.scatter_reduce_(0, state_of[cols], q, how)
        new = torch.clamp(best, max=1.0) if reward is None else reward + case["discount"] * best
        new = torch.where(mask == 1, 1.0, torch.where(mask == 2, 0.0, new))
        new = torch.where(hor > k, new, V)
        residual = torch.where(hor > k, new - V, residual)
        V = new
        if case["infinite"] and float(residual.abs().max()) < case["tol"]:
            break
    out = dict(V=V, k=None)
    if case["path"] not in ("batch", "served"):
        # a query that has settled ends on differences of rounding, which no other arithmetic repeats
        settled = float(residual.abs().max()) < 1e-9
        out.update(residual=None if settled else residual, policy=None)
    return out
