"""Which kernel a step call takes: the shapes by which the resident and the grid
kernel are tested do run on them, so a rule or a plan that sends one elsewhere
shows up here."""
import json
import time

import numpy as np
import pytest
import torch

import paper_2401_04068_gb300 as g
from test_resident_gpu import GRID, _lengths, _run, _same
from workloads import banded_batch, banded_imdp, random_imdp
from workloads.imdp_synth import concat_block_diagonal

pytestmark = pytest.mark.gpu


def _route(models, specs, n, **launch):
    sess = g.imdp_session_create(models, specs)
    if launch:
        g.imdp_session_set_launch(sess, **launch)
    r = g.imdp_session_step_route(sess, n)
    sess.close()
    return r


def _alone(m, n=20, dtype=g.IMDP_F64, **kw):
    model = g.create_model(m, dtype=dtype)
    r = _route([model], [g.make_spec(horizon=20, reach=m.goal, **kw)], n)
    model.close()
    return r


@pytest.mark.parametrize("dtype", [g.IMDP_F64, g.IMDP_F32])
def test_kernels_of_one_problem(dtype):
    for lens, kernel in (((1, 2, 7, 8, 9), g.KERNEL_RESIDENT), ((31, 32, 33, 63, 64, 65), g.KERNEL_RESIDENT),
                         ((255, 256, 257, 300), g.KERNEL_GRID), ((5,), g.KERNEL_RESIDENT)):
        r = _alone(_lengths(1100, lens, 5), dtype=dtype)
        assert (r["kernel"], r["launches"], r["copied"]) == (kernel, 1, 1), lens
    for name in GRID:
        r = _alone(GRID[name](), dtype=dtype)
        assert (r["kernel"], r["launches"], r["threads"]) == (g.KERNEL_GRID, 1, 768), name
        assert r["group"] == (8 if name == "sink" else 32) and r["copied"] == (name not in ("long_sink", "wide")), name
    for n, a, k in ((5, 1, 5), (7, 3, 4), (64, 1, 12), (330, 3, 4), (1000, 1, 3)):
        r = _alone(banded_imdp(n, a, n * a * (min(k, n) + 1) + 1, eps=0.1, seed=n), dtype=dtype)
        assert r["kernel"] == g.KERNEL_RESIDENT and r["units"] == 1 and r["copied"] == 1, n
        assert (r["cluster"] == 1) == (n == 5), n
    # (the sink is a state more)
    for n, a, finite, infinite in ((1, 1, 3, 3), (4, 1, 3, 3), (4, 2, 5, 3), (5, 1, 5, 5), (4, 5, 5, 5)):
        m = banded_imdp(n, a, n * a * (min(2, n) + 1) + 1, eps=0.1, seed=n)
        assert _alone(m, dtype=dtype)["kernel"] == finite, (n, a)
        assert _alone(m, dtype=dtype, infinite_time=True, eps=1e-6)["kernel"] == infinite, (n, a)
    for a, threads in ((1, 384), (3, 768)):
        r = _alone(banded_imdp(610, a, 610 * a * 21 + 610 * a + 1, eps=0.1, seed=31), dtype=dtype)
        assert (r["kernel"], r["cluster"], r["threads"]) == (g.KERNEL_RESIDENT, 16, threads)


def test_kernels_of_many_problems():
    ms = [banded_imdp(20 + 7 * (i % 60), 1 + i % 3, (20 + 7 * (i % 60)) * (1 + i % 3) * (3 + i % 17) + 1, seed=100 + i)
          for i in range(200)]
    models = [g.create_model(x) for x in ms]
    specs = [g.make_spec(horizon=30, reach=x.goal) for x in ms]
    r = _route(models, specs, 30)
    assert r["kernel"] == g.KERNEL_RESIDENT and r["units"] == 200 and r["threads"] == 384 and r["ctas"] > 152
    # short calls and explicit configurations run one launch an iteration
    assert _route(models, specs, 3)["launches"] == 3
    assert _route(models, specs, 30, kernel=g.KERNEL_RING) == dict(kernel=g.KERNEL_RING, launches=30, units=0,
                                                                  cluster=0, ctas=0, threads=0, group=0, copied=0)
    m = concat_block_diagonal([banded_batch(40, 60, 1, 60 * 12 + 60 + 1, seed=3), random_imdp(1, seed=4),
                               banded_imdp(330, 1, 330 * 70 + 330 + 1, seed=5),
                               random_imdp(37, max_actions=1, seed=6)])
    model = g.create_model(m)
    finite, infinite = g.make_spec(horizon=30, reach=m.goal), g.make_spec(infinite_time=True, horizon=50, reach=m.goal)
    r = _route([model], [finite], 30)
    assert r["kernel"] == g.KERNEL_RESIDENT and r["units"] > 40 and r["cluster"] > 1
    assert _route([model], [infinite], 30)["units"] == 1


# more parts than two CTAs on every SM hold, in CTAs of half the threads; rounds of them, the last one not full
@pytest.mark.parametrize("storage", [g.IMDP_F64, g.IMDP_F32])
@pytest.mark.parametrize("blocks", [304, 1001])
def test_parts_on_half_size_ctas(storage, blocks):
    m = banded_batch(blocks, 40, 2, 40 * 2 * 11 + 40 * 2 + 1, eps=0.1, seed=blocks)
    model = g.create_model(m, dtype=storage)
    specs = [g.make_spec(horizon=25, reach=m.goal)]
    r = _route([model], specs, 25)
    assert (r["kernel"], r["units"], r["cluster"], r["threads"], r["ctas"]) == (g.KERNEL_RESIDENT, blocks, 1, 384, 304)
    _same(_run([model], [m], specs, g.KERNEL_RING, policy=True), _run([model], [m], specs, g.KERNEL_RULE, policy=True))
    model.close()


def test_bad_route_queries():
    m = random_imdp(5, seed=1)
    model = g.create_model(m)
    sess = g.imdp_session_create([model], [g.make_spec(horizon=3, reach=m.goal)])
    with pytest.raises(g.ImdpError):
        g.imdp_session_step_route(sess, 0)
    sess.close()
    model.close()


@pytest.mark.parametrize("storage", [g.IMDP_F64, g.IMDP_F32])
def test_requests_share_launches(storage):
    ms = [banded_imdp(2000, 2, 2000 * 2 * 150 + 2001, eps=0.1, seed=70), banded_imdp(6000, 3, 6000 * 3 * 3 + 1, seed=71),
          banded_imdp(70, 2, 70 * 2 * 9 + 1, seed=75)]
    models = [g.create_model(m, dtype=storage) for m in ms]
    for launch in ({}, dict(kernel=g.KERNEL_RING)):
        server = g.imdp_server_create(256 << 20)
        if launch:
            g.imdp_server_set_launch(server, **launch)
        tickets = [g.imdp_server_submit(server, models[i % 3], g.make_spec(horizon=60 + i, reach=ms[i % 3].goal))
                   for i in range(12)]
        for i, t in enumerate(tickets):
            assert g.imdp_server_wait(server, t, 60000.0, np.zeros(ms[i % 3].n_states)) == g.IMDP_OK
        time.sleep(0.2)  # the worker counts a launch after its requests have retired
        n = g.imdp_server_launches(server)
        assert (n["shared"] > 0, n["per_iteration"] > 0) == ((False, True) if launch else (True, False)), n
        assert n["shared"] + n["per_iteration"] // 8 == g.imdp_server_stats(server)["chunks"]
        server.close()


@pytest.mark.parametrize("field", ["cta_warps", "ctas_per_sm", "tile_entries", "wide_col"])
def test_a_partial_configuration_shapes_the_steps(field):
    # kernel 0 with a field given: the per-iteration kernels run in that shape, as
    # imdp_session_get_launch reports; all zero goes back to the rule
    value = dict(cta_warps=24, ctas_per_sm=3, tile_entries=600, wide_col=200)[field]
    m = banded_imdp(2000, 1, 2000 * 40 + 2000 + 1, eps=0.05, seed=82)
    model = g.create_model(m)
    spec = g.make_spec(horizon=30, reach=m.goal)
    sess = g.imdp_session_create([model], [spec])
    assert g.imdp_session_step_route(sess, 30)["kernel"] in (g.KERNEL_RESIDENT, g.KERNEL_GRID)
    g.imdp_session_set_launch(sess, **{field: value})
    r, got = g.imdp_session_step_route(sess, 30), g.imdp_session_get_launch(sess)
    assert r["kernel"] == got["kernel"] == g.KERNEL_RING and r["launches"] == 30
    assert field == "ctas_per_sm" or got[field] == value
    g.imdp_session_step(sess, 30)
    raw, _ = g.imdp_session_checkpoint(sess, 0)
    g.imdp_session_set_launch(sess)
    assert g.imdp_session_step_route(sess, 30)["kernel"] in (g.KERNEL_RESIDENT, g.KERNEL_GRID)
    g.imdp_session_reset(sess)
    g.imdp_session_step(sess, 30)
    np.testing.assert_array_equal(raw, g.imdp_session_checkpoint(sess, 0)[0])
    sess.close()
    server = g.imdp_server_create(64 << 20)
    g.imdp_server_set_launch(server, **{field: value})
    t = g.imdp_server_submit(server, model, spec)
    assert g.imdp_server_wait(server, t, 60000.0, np.zeros(m.n_states)) == g.IMDP_OK
    time.sleep(0.2)
    assert g.imdp_server_launches(server)["shared"] == 0
    server.close()
    model.close()


def test_autotuned_sessions_keep_the_faster_rule(tmp_path):
    # The rule's own kernels are among the candidates: a tuned session is no slower
    # than an untuned one. 64 parts of 120 states take the resident kernel by rule.
    m = banded_batch(64, 120, 1, 120 * 30 + 120 + 1, eps=0.05, seed=7)
    model = g.create_model(m)
    spec = g.make_spec(horizon=60, reach=m.goal)
    cache = tmp_path / "tuned.json"

    def tuned(iters=60):
        sess = g.imdp_session_create([model], [spec])
        cfg, ms = g.imdp_session_autotune(sess, iters, str(cache))
        return sess, cfg, ms

    sess, cfg, ms = tuned()
    # (this query per iteration takes about 10 us an iteration at best, by rule about 3)
    assert g.imdp_session_step_route(sess, 60)["kernel"] == g.KERNEL_RESIDENT
    assert cfg["kernel"] in (g.KERNEL_RING, g.KERNEL_DIRECT, g.KERNEL_SLICE) and ms > 0
    assert cfg["kernel"] == g.imdp_session_get_launch(sess)["kernel"] == g.imdp_session_step_route(sess, 1)["kernel"]
    g.imdp_session_run(sess)
    raw, k = g.imdp_session_checkpoint(sess, 0)
    sess.close()
    assert k == 60
    plain = g.imdp_session_create([model], [spec])
    g.imdp_session_run(plain)
    np.testing.assert_array_equal(raw, g.imdp_session_checkpoint(plain, 0)[0])
    plain.close()
    # the cached choice: the same, without timing
    sess, cfg2, ms = tuned()
    assert ms == 0.0 and cfg2 == cfg and g.imdp_session_step_route(sess, 60)["kernel"] == g.KERNEL_RESIDENT
    sess.close()
    # an entry that knows nothing of the rule's kernels is timed against them once
    data = json.loads(cache.read_text())
    entry = next(iter(data.values()))
    assert entry.pop("long_by_rule") == 1
    cache.write_text(json.dumps(data).replace("}, ", "},\n"))
    sess, cfg3, ms = tuned()
    assert ms > 0 and cfg3 == cfg and g.imdp_session_step_route(sess, 60)["kernel"] == g.KERNEL_RESIDENT
    sess.close()
    assert next(iter(json.loads(cache.read_text()).values()))["long_by_rule"] == 1
    # tuned on single iterations: the same
    cache.unlink()
    sess, _, _ = tuned(1)
    assert g.imdp_session_step_route(sess, 60)["kernel"] == g.KERNEL_RESIDENT
    sess.close()
    model.close()


# parts on either side of the shared memory that each of two CTAs of an SM can have
@pytest.mark.parametrize("storage", [g.IMDP_F64, g.IMDP_F32])
@pytest.mark.parametrize("states,threads,ctas", [(1000, 384, 304), (1300, 768, 152)])
def test_half_size_ctas_only_where_two_fit_an_sm(storage, states, threads, ctas):
    m = banded_batch(310, states, 1, states * 4 + 1, eps=0.1, seed=states)
    model = g.create_model(m, dtype=storage)
    specs = [g.make_spec(horizon=12, reach=m.goal)]
    r = _route([model], specs, 12)
    assert (r["kernel"], r["units"], r["cluster"], r["threads"], r["ctas"]) == (g.KERNEL_RESIDENT, 310, 1, threads, ctas)
    _same(_run([model], [m], specs, g.KERNEL_RING), _run([model], [m], specs, g.KERNEL_RULE))
    model.close()


# one large unit beside small ones: its cluster alone would take longer than the whole GPU does
@pytest.mark.parametrize("as_parts", [True, False])
def test_a_dominant_unit_takes_the_whole_gpu(as_parts):
    ms = [banded_imdp(2000, 2, 2000 * 2 * 1251 + 1, eps=0.1, seed=1)]
    ms += [banded_imdp(200, 1, 200 * 21 + 1, eps=0.1, seed=2 + i) for i in range(12)]
    if as_parts:
        ms = [concat_block_diagonal(ms)]
    models = [g.create_model(m) for m in ms]
    specs = [g.make_spec(horizon=12, reach=m.goal) for m in ms]
    kernel = _route(models, specs, 12)["kernel"]
    assert kernel == g.KERNEL_GRID if as_parts else kernel not in (g.KERNEL_GRID, g.KERNEL_RESIDENT)
    _same(_run(models, ms, specs, g.KERNEL_RING), _run(models, ms, specs, g.KERNEL_RULE))
    for m in models:
        m.close()


def test_a_long_horizon_counts_in_the_choice():
    # one problem with a long horizon beside 40 small ones with a short one: most of the
    # time its cluster would run alone, which pays for 300,000 transitions only
    small = banded_imdp(400, 1, 400 * 201 + 1, eps=0.1, seed=2)
    for n, k, K, resident in ((700, 450, 200, True), (1000, 990, 500, False)):
        ms = [banded_imdp(n, 1, n * (k + 1) + 1, eps=0.1, seed=1)] + [small] * 40
        models = [g.create_model(m) for m in ms]
        specs = [g.make_spec(horizon=20 if i else K, reach=m.goal) for i, m in enumerate(ms)]
        assert (_route(models, specs, K)["kernel"] == g.KERNEL_RESIDENT) == resident, n
        for m in models:
            m.close()


# units a few more than clusters of 16 (7 fit the GPU) or 8 CTAs (15): smaller clusters, all at once
@pytest.mark.parametrize("n", [4, 8, 20])
@pytest.mark.parametrize("storage", [g.IMDP_F64, g.IMDP_F32])
def test_every_unit_has_a_cluster(n, storage):
    one = banded_imdp(400, 1, 400 * 201 + 1, eps=0.1, seed=5)
    m = concat_block_diagonal([one] * n)
    model = g.create_model(m, dtype=storage)
    specs = [g.make_spec(horizon=12, reach=m.goal)]
    r = _route([model], specs, 12)
    assert (r["kernel"], r["units"], r["ctas"]) == (g.KERNEL_RESIDENT, n, n * r["cluster"]) and r["cluster"] > 1
    _same(_run([model], [m], specs, g.KERNEL_RING), _run([model], [m], specs, g.KERNEL_RULE))
    model.close()


# a state or a few that nothing connects to the model, before, behind and between: they count as part of it
@pytest.mark.parametrize("where", ["behind", "before", "both", "several"])
@pytest.mark.parametrize("shape", [(5, 5), (240, 108), (960, 559)])
def test_detached_states_are_no_unit_of_their_own(shape, where):
    n, k = shape
    body = banded_imdp(n, 1, n * (k + 1) + 1, eps=0.1, seed=1)
    dot = random_imdp(1, 1, 1, seed=2)
    m = concat_block_diagonal({"behind": [body, dot], "before": [dot, body], "both": [dot, body, dot],
                               "several": [dot, dot, body, dot, dot, dot]}[where])
    model, alone = g.create_model(m), _alone(body)
    specs = [g.make_spec(horizon=20, reach=m.goal)]
    r = _route([model], specs, 20)
    assert (r["kernel"], r["units"], r["copied"]) == (alone["kernel"], 1, 1)
    _same(_run([model], [m], specs, g.KERNEL_RING, policy=True), _run([model], [m], specs, g.KERNEL_RULE, policy=True))
    model.close()


# how long one launch of a long step call holds the GPU: about 10 ms, about 100 where the
# units do not all run at once (four times that, as the estimate is one of a cost model)
@pytest.mark.parametrize("shape,n,bound", [("small", 40000, 0.04), ("large", 12000, 0.04), ("rounds", 2000, 0.4)])
def test_launches_are_bounded(shape, n, bound):
    m = {"small": lambda: banded_imdp(240, 1, 240 * 109 + 1, eps=0.1, seed=1),
         "large": lambda: banded_imdp(960, 1, 960 * 560 + 1, eps=0.1, seed=1),
         "rounds": lambda: banded_batch(1000, 200, 1, 200 * 101 + 1, eps=0.1, seed=1)}[shape]()
    model = g.create_model(m)
    sess = g.imdp_session_create([model], [g.make_spec(horizon=n, reach=m.goal)])
    r = g.imdp_session_step_route(sess, n)
    assert r["kernel"] == (g.KERNEL_GRID if shape == "large" else g.KERNEL_RESIDENT)
    g.imdp_session_step(sess, 4)
    torch.cuda.synchronize()
    t = time.perf_counter()
    g.imdp_session_step(sess, n - 4)
    torch.cuda.synchronize()
    seconds = (time.perf_counter() - t) / g.imdp_session_step_route(sess, n - 4)["launches"]
    assert seconds <= bound, (seconds, r)
    sess.close()
    model.close()


# few, very long columns on 32-bit storage whose bounds are mostly kept exact: the
# per-iteration kernels are the faster ones there
@pytest.mark.parametrize("n,k,grid", [(3840, 2227, False), (3000, 1500, True)])
def test_long_exact_columns_stay_per_iteration(n, k, grid):
    m = banded_imdp(n, 1, n * (k + 1) + 1, eps=0.1, seed=1)
    model = g.create_model(m, dtype=g.IMDP_F32)
    exact = g.imdp_model_exact_columns(model)[1] / m.nnz
    spec = g.make_spec(horizon=100, reach=m.goal)
    kernel = _route([model], [spec], 100)["kernel"]
    assert (kernel == g.KERNEL_GRID) == grid and exact > (0.6 if grid else 0.8), exact
    wide = g.create_model(m)
    assert _route([wide], [spec], 100)["kernel"] == g.KERNEL_GRID  # on 64-bit storage
    wide.close()

    def seconds(**launch):
        sess = g.imdp_session_create([model], [spec])
        if launch:
            g.imdp_session_set_launch(sess, **launch)
        best = 1.0
        for _ in range(4):
            g.imdp_session_reset(sess)
            torch.cuda.synchronize()
            t = time.perf_counter()
            g.imdp_session_step(sess, 100)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        sess.close()
        return best

    # the rule's choice is no slower than the kernel it took before there was a grid kernel
    assert seconds() <= 1.08 * seconds(kernel=g.KERNEL_DIRECT, ctas_per_sm=3, tile_entries=1024)
    model.close()


def test_launches_are_bounded_beside_a_long_horizon():
    # 2,000 problems of 300 iterations and one of 20,000: the launch that runs them all
    # is no longer than others, although an average iteration takes next to nothing
    small = banded_imdp(200, 1, 200 * 101 + 1, eps=0.1, seed=3)
    model = g.create_model(small)
    n = 2001
    specs = [g.make_spec(horizon=20000 if i == 0 else 300, reach=small.goal) for i in range(n)]
    sess = g.imdp_session_create([model] * n, specs)
    r = g.imdp_session_step_route(sess, 20000)
    assert r["kernel"] == g.KERNEL_RESIDENT
    # (40 million transitions take 0.12 ms an iteration at the resident kernel's rate; twice the usual 0.1 s)
    assert 20000 / r["launches"] <= 2 * 0.1 / 0.12e-3, r
    sess.close()
    model.close()


# few iterations, most of them with nearly every column to settle: long columns stay per
# iteration, and a cluster of 16 SMs is left for the whole GPU
@pytest.mark.parametrize("n,k,short,long,kernels", [
    (3840, 2240, 63, 64, (g.KERNEL_DIRECT, g.KERNEL_GRID)), (3000, 1700, 31, 32, (g.KERNEL_DIRECT, g.KERNEL_GRID)),
    (1500, 80, 23, 24, (g.KERNEL_GRID, g.KERNEL_RESIDENT))])
def test_few_iterations_of_long_searches(n, k, short, long, kernels):
    m = banded_imdp(n, 1, n * (k + 1) + 1, eps=0.1, seed=1)
    model = g.create_model(m)
    for kw, want in ((dict(horizon=short), 0), (dict(horizon=long), 1),
                     (dict(infinite_time=True, eps=1e-6, horizon=10), 1)):
        assert _route([model], [g.make_spec(reach=m.goal, **kw)], 10)["kernel"] == kernels[want], kw
    model.close()
