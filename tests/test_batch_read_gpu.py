"""A batch's results read in one pass: the same doubles, counts and status as
each problem's own session, into host, device and overlapping outputs."""
import numpy as np
import pytest
import torch

import paper_2401_04068_gb300 as g
from workloads import random_imdp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["host", "device", "mixed", "overlap", "noconv"])
def test_batch_results(kind):
    rng = np.random.default_rng(2)
    ms = [random_imdp(n, 2, 6, seed=n) for n in (7, 1, 300, 64, 33)]
    models = [g.create_model(m) for m in ms]
    kws = [dict(horizon=3 + i, reach=m.goal) for i, m in enumerate(ms)]
    kws[2] = dict(property=g.IMDP_REWARD, horizon=9, reward=rng.uniform(-2, 3, 300), discount=0.9)
    kws[3] = dict(horizon=0, reach=ms[3].goal)
    if kind == "noconv":
        kws[4] = dict(infinite_time=True, eps=1e-12, horizon=2, reach=ms[4].goal)
    specs = [g.make_spec(**kw) for kw in kws]
    want = []
    for model, m, spec in zip(models, ms, specs):
        sess = g.imdp_session_create([model], [spec])
        g.imdp_session_run(sess)
        V, k = np.zeros(m.n_states), [0]
        g.imdp_session_read(sess, 0, V, k, None, None, check=False)
        sess.close()
        want.append((V, k[0]))
    outs = [np.full(m.n_states, -1.0) for m in ms]
    if kind in ("device", "mixed"):
        outs = [torch.full((m.n_states,), -1.0, dtype=torch.float64, device="cuda")
                if kind == "device" or i % 2 else outs[i] for i, m in enumerate(ms)]
    if kind == "overlap":
        shared = np.full(300, -1.0)
        outs = [shared[:m.n_states] for m in ms]
    ks = [0] * len(ms)
    st = g.imdp_value_iteration_batch(models, specs, outs, ks)
    assert st == (g.IMDP_ENOCONV if kind == "noconv" else g.IMDP_OK)
    assert ks == [k for _, k in want]
    if kind == "overlap":  # one problem after the other: the last ones stand
        expect = want[2][0].copy()
        expect[:64] = want[3][0]
        expect[:33] = want[4][0]
        np.testing.assert_array_equal(shared, expect)
        return
    for o, (V, _) in zip(outs, want):
        np.testing.assert_array_equal(o.cpu().numpy() if torch.is_tensor(o) else o, V)
