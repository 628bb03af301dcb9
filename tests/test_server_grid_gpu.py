"""Requests that share launches of the grid kernel: several CTAs to a large one,
small ones behind one another on one CTA, arrivals while others run, budgets that
leave the plan no room. Every result equals the request's own query by the
per-iteration ring kernel."""
import time

import numpy as np
import pytest

import paper_2401_04068_gb300 as g
from workloads import banded_imdp, random_imdp

pytestmark = pytest.mark.gpu


def _alone(model, m, spec):
    sess = g.imdp_session_create([model], [spec])
    g.imdp_session_set_launch(sess, kernel=g.KERNEL_RING)
    g.imdp_session_run(sess)
    V, k = np.zeros(m.n_states), [0]
    st = g.imdp_session_read(sess, 0, V, k, None, None, check=False)
    sess.close()
    return st, V, k[0]


@pytest.mark.parametrize("storage", ["f64", "f32", "both"])
@pytest.mark.parametrize("budget", ["ample", "tight"])
def test_requests_sharing_the_grid(storage, budget):
    ms = [banded_imdp(2000, 2, 2000 * 2 * 150 + 2001, eps=0.1, seed=70), banded_imdp(6000, 3, 6000 * 3 * 3 + 1, seed=71),
          random_imdp(1, 1, 1, seed=72), banded_imdp(300, 1, 300 * 280 + 1, seed=73), random_imdp(50, 3, 0.5, seed=74),
          banded_imdp(70, 2, 70 * 2 * 9 + 1, seed=75)]
    dt = [g.IMDP_F64 if storage == "f64" or (storage == "both" and i % 2) else g.IMDP_F32 for i in range(len(ms))]
    models = [g.create_model(m, dtype=d) for m, d in zip(ms, dt)]
    reqs = []
    for i in range(26):
        j = i % len(ms)
        m = ms[j]
        kw = dict(horizon=(20 + 7 * i) % 60, reach=m.goal, pessimistic=i % 3 != 0, maximize=i % 4 != 1)
        if i % 5 == 3:
            kw.update(infinite_time=True, eps=1e-4, horizon=(2, 400)[i % 2])
        if i % 7 == 4:
            kw = dict(property=g.IMDP_REWARD, horizon=15, reward=np.linspace(-1, 1, m.n_states), discount=0.9)
        reqs.append((j, g.make_spec(**kw)))
    want = [_alone(models[j], ms[j], s) for j, s in reqs]
    # tight: the largest request and little more, so the miss lists find no room beside some mixes
    most = max(25 * m.n_states + 4 * int(m.stateptr[-1]) + 16 * m.n_states for m in ms)
    server = g.imdp_server_create((256 << 20) if budget == "ample" else max(1 << 20, int(1.2 * most)))
    tickets = []
    for i, (j, spec) in enumerate(reqs):
        tickets.append(g.imdp_server_submit(server, models[j], spec))
        if i in (5, 13, 14):
            time.sleep(0.003)
    for (j, _), t, (st, V, k) in zip(reqs, tickets, want):
        out, ko = np.zeros(ms[j].n_states), [0]
        assert g.imdp_server_wait(server, t, 60000.0, out, ko) == st
        assert ko[0] == k
        np.testing.assert_array_equal(out, V)
    server.close()
