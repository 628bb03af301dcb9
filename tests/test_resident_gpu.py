"""The resident and grid kernels (by rule, several iterations in one launch)
against the per-iteration ring kernel: the same words, iteration counts,
residuals and policies, at the sizes where their tiling can go wrong."""
import numpy as np
import pytest

import paper_2401_04068_gb300 as g
from gpu_helpers import TOL_F64, run_oracle
from workloads import banded_batch, banded_imdp, random_imdp
from workloads.imdp_synth import IMDPInput, concat_block_diagonal

pytestmark = pytest.mark.gpu


def _run(models, ms, specs, kernel, steps=None, policy=False):
    sess = g.imdp_session_create(models, specs, want_policy=[1] * len(ms) if policy else None)
    g.imdp_session_set_launch(sess, kernel=kernel)
    if steps is None:
        g.imdp_session_run(sess)
    else:
        for n in steps:
            g.imdp_session_step(sess, n)
    out = []
    for i, m in enumerate(ms):
        raw, k = g.imdp_session_checkpoint(sess, i)
        res = np.zeros(m.n_states)
        pol = np.zeros((k, m.n_states), np.int32) if policy else None
        g.imdp_session_read(sess, i, None, None, res, pol, check=False)
        out.append((raw, k, res, pol))
    sess.close()
    return out


def _same(a, b):
    for (ra, ka, sa, pa), (rb, kb, sb, pb) in zip(a, b):
        assert ka == kb
        np.testing.assert_array_equal(ra, rb)
        np.testing.assert_array_equal(sa, sb)
        if pa is not None:
            np.testing.assert_array_equal(pa, pb)


def _lengths(n, lens, seed, wide=False):
    """One action per state; column j has lens[j % len(lens)] entries at scattered states."""
    rng = np.random.default_rng(seed)
    colptr, rows, lo, up = [0], [], [], []
    for s in range(n):
        k = lens[s % len(lens)]
        r = np.sort(rng.choice(n, k, replace=False))
        p = rng.random(k) + 0.05
        p /= p.sum()
        rows.append(r)
        lo.append(np.zeros(k) if wide else p * (1 - 0.3 * rng.random(k)))
        up.append(np.ones(k) if wide else np.minimum(1, p * (1 + 0.3 * rng.random(k))))
        colptr.append(colptr[-1] + k)
    return IMDPInput(n, np.arange(n + 1, dtype=np.int32), np.array(colptr, np.int32),
                     np.concatenate(rows).astype(np.int32), np.concatenate(lo), np.concatenate(up),
                     np.arange(n // 2, n // 2 + 3, dtype=np.int32))


# column lengths around the lane groups (8 and 32 lanes), their batches of trips and the search's chunks
@pytest.mark.parametrize("lens", [(1, 2, 7, 8, 9), (31, 32, 33, 63, 64, 65), (255, 256, 257, 300), (5,)])
@pytest.mark.parametrize("pess", [True, False])
@pytest.mark.parametrize("dtype", ["f64", "f32", "f32_exact", "wide"])
def test_column_lengths(lens, pess, dtype):
    m = _lengths(1100, lens, 5, wide=dtype == "wide")
    if dtype.startswith("f32"):
        model = g.create_model(m, dtype=g.IMDP_F32, budget=1.2e-9 if dtype == "f32_exact" else 1.0)
    else:
        model = g.create_model(m)
    spec = [g.make_spec(horizon=20, reach=m.goal, pessimistic=pess)]
    ref = _run([model], [m], spec, g.KERNEL_RING)
    _same(ref, _run([model], [m], spec, g.KERNEL_RULE))
    _same(ref, _run([model], [m], spec, g.KERNEL_RULE, steps=(4, 1, 9, 30)))  # past the horizon too
    model.close()


@pytest.mark.parametrize("case", ["reach_avoid", "reward", "infinite", "cap"])
@pytest.mark.parametrize("actions", [1, 3])
def test_properties_and_policies(case, actions):
    m = banded_imdp(610, actions, 610 * actions * 21 + 610 * actions + 1, eps=0.1, seed=31)
    model = g.create_model(m)
    kw = dict(horizon=25, reach=m.goal)
    if case == "reach_avoid":
        kw.update(property=g.IMDP_REACH_AVOID, avoid=np.setdiff1d(np.arange(0, 611, 13), m.goal), pessimistic=False)
    elif case == "reward":
        kw = dict(property=g.IMDP_REWARD, horizon=25, reward=np.linspace(-1, 2, 611), discount=0.9, maximize=False)
    elif case == "infinite":
        kw = dict(infinite_time=True, eps=1e-8, horizon=3000, reach=m.goal)
    elif case == "cap":
        kw = dict(infinite_time=True, eps=1e-300, horizon=37, reach=m.goal)
    spec = [g.make_spec(**kw)]
    policy = not kw.get("infinite_time")
    _same(_run([model], [m], spec, g.KERNEL_RING, policy=policy), _run([model], [m], spec, g.KERNEL_RULE, policy=policy))
    model.close()


@pytest.mark.parametrize("dtype", [g.IMDP_F64, g.IMDP_F32])
def test_parts_of_one_model(dtype):
    # blocks that no transition leaves, of different sizes (one state among
    # them), run as parts; the last boundary is the model's end
    blocks = [banded_batch(40, 60, 1, 60 * 12 + 60 + 1, seed=3), random_imdp(1, seed=4),
              banded_imdp(330, 1, 330 * 70 + 330 + 1, seed=5), random_imdp(37, max_actions=1, seed=6)]
    m = concat_block_diagonal(blocks)
    model = g.create_model(m, dtype=dtype)
    for kw in (dict(horizon=30), dict(horizon=0), dict(infinite_time=True, eps=1e-7, horizon=5000)):
        spec = [g.make_spec(reach=m.goal, **kw)]
        policy = kw.get("horizon") == 30
        _same(_run([model], [m], spec, g.KERNEL_RING, policy=policy),
              _run([model], [m], spec, g.KERNEL_RULE, policy=policy))
    if dtype == g.IMDP_F64:
        st, V, _, _, _ = g.value_iteration(model, m.n_states, horizon=30, reach=m.goal)
        _, oV, _, _, _ = run_oracle(m, horizon=30, reach=m.goal)
        np.testing.assert_allclose(V, oV, rtol=0, atol=TOL_F64)
    model.close()


def test_batch_of_uneven_problems():
    # more units than clusters, horizons 0 and 1 among them, infinite horizons
    # beside finite ones, both adversaries
    ms = [banded_imdp(20 + 7 * (i % 60), 1 + i % 3, (20 + 7 * (i % 60)) * (1 + i % 3) * (3 + i % 17) + 1, seed=100 + i)
          for i in range(200)]
    models = [g.create_model(x) for x in ms]
    specs = [g.make_spec(infinite_time=True, eps=1e-6, horizon=400, reach=x.goal) if i % 50 == 7 else
             g.make_spec(horizon=i % 33, reach=x.goal, pessimistic=i % 2 == 0, maximize=i % 5 != 0)
             for i, x in enumerate(ms)]
    _same(_run(models, ms, specs, g.KERNEL_RING), _run(models, ms, specs, g.KERNEL_RULE))
    for x in models:
        x.close()


# one problem of the whole GPU: windows with a far last destination (the sink) or
# the whole state space, columns around the lane groups and beyond one tile,
# many misses at once (listed for all CTAs), entries copied to shared memory or not
GRID = {
    "sink": lambda: banded_imdp(6000, 3, 6000 * 3 * 41 + 6000 * 3 + 1, eps=0.1, seed=11),
    "long_sink": lambda: banded_imdp(5000, 1, 5000 * 390 + 5000 + 1, eps=0.1, seed=12),
    "scattered": lambda: _lengths(3001, (60, 61, 190, 256, 257, 31), 13),
    "wide": lambda: _lengths(2100, (1279, 1280, 1281, 40, 1900), 14),
    "loose": lambda: _lengths(2500, (90, 200, 33), 15, wide=True),
    # few columns to a CTA: its misses are settled by teams of warps
    "few_long": lambda: _lengths(900, (500, 700, 333, 899), 16),
    "few_loose": lambda: _lengths(700, (640, 321), 17, wide=True),
}


@pytest.mark.parametrize("shape", sorted(GRID))
@pytest.mark.parametrize("case", ["reach", "optimistic_avoid", "reward", "infinite", "f32", "f32_exact"])
def test_one_large_problem(shape, case):
    m = GRID[shape]()
    if case.startswith("f32"):
        model = g.create_model(m, dtype=g.IMDP_F32, budget=1.0 if case == "f32" else 2e-9)
    else:
        model = g.create_model(m)
    kw = dict(horizon=18, reach=m.goal)
    if case == "optimistic_avoid":
        kw.update(property=g.IMDP_REACH_AVOID, avoid=np.setdiff1d(np.arange(0, m.n_states, 17), m.goal),
                  pessimistic=False, maximize=False)
    elif case == "reward":
        r = np.random.default_rng(3).uniform(-1, 1, m.n_states)
        kw = dict(property=g.IMDP_REWARD, horizon=18, reward=r, discount=0.95)
    elif case == "infinite":
        kw = dict(infinite_time=True, eps=1e-4, horizon=60, reach=m.goal)
    spec = [g.make_spec(**kw)]
    policy = case in ("reach", "reward")
    ref = _run([model], [m], spec, g.KERNEL_RING, policy=policy)
    _same(ref, _run([model], [m], spec, g.KERNEL_RULE, policy=policy))
    if case == "reach":
        _same(ref, _run([model], [m], spec, g.KERNEL_RULE, steps=(5, 2, 4, 20), policy=True))
        _, oV, _, _, _ = run_oracle(m, **kw)
        assert float(np.max(np.abs(ref[0][0].astype(np.float64) / 2.0 ** 63 - oV))) <= TOL_F64
    model.close()


# the smallest problems (one CTA, half its warps, or a few CTAs) and step calls
# too short for a resident launch in between (the single-CTA kernel)
@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 1, 5), (7, 3, 4), (64, 1, 12), (330, 3, 4), (1000, 1, 3)])
@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_small_problem(shape, storage):
    n, a, k = shape
    m = banded_imdp(n, a, n * a * (min(k, n) + 1) + 1, eps=0.1, seed=n)
    model = g.create_model(m, dtype=g.IMDP_F32 if storage == "f32" else g.IMDP_F64)
    for kw in (dict(horizon=23, reach=m.goal), dict(infinite_time=True, eps=1e-5, horizon=90, reach=m.goal),
               dict(horizon=23, reach=m.goal, pessimistic=False, maximize=False)):
        spec = [g.make_spec(**kw)]
        policy = "infinite_time" not in kw
        ref = _run([model], [m], spec, g.KERNEL_RING, policy=policy)
        _same(ref, _run([model], [m], spec, g.KERNEL_RULE, policy=policy))
        _same(ref, _run([model], [m], spec, g.KERNEL_RULE, steps=(3, 5, 1, 4, 2, 90), policy=policy))
    model.close()
