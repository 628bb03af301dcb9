"""Requests that share one CTA of the server's launches all get on: requests of an
infinite horizon that converge slowly do not hold up finite ones behind them."""
import numpy as np
import pytest

import paper_2401_04068_gb300 as g
from workloads import banded_imdp

pytestmark = pytest.mark.gpu


def test_slow_infinite_requests_hold_up_nobody():
    # the long request sets the length of the plan, so that all small ones are
    # put behind one another on one CTA
    wide = banded_imdp(2000, 2, 2000 * 2 * 150 + 1, eps=0.1, seed=1)
    small = banded_imdp(600, 1, 600 * 31 + 1, eps=0.1, seed=2)
    mw, ms = g.create_model(wide), g.create_model(small)
    slow = g.make_spec(property=g.IMDP_REWARD, infinite_time=True, eps=1e-12, horizon=60000, discount=0.99999,
                       reward=np.linspace(0, 1, small.n_states))
    finite = [g.make_spec(horizon=250 + 10 * i, reach=small.goal) for i in range(3)]
    server = g.imdp_server_create(256 << 20)
    long = g.imdp_server_submit(server, mw, g.make_spec(horizon=300000, reach=wide.goal))
    slows = [g.imdp_server_submit(server, ms, slow) for _ in range(3)]
    tickets = [g.imdp_server_submit(server, ms, f) for f in finite]
    for i, t in enumerate(tickets):
        V, k = np.zeros(small.n_states), [0]
        assert g.imdp_server_wait(server, t, 60000.0, V, k) == g.IMDP_OK and k[0] == 250 + 10 * i
        sess = g.imdp_session_create([ms], [finite[i]])
        g.imdp_session_set_launch(sess, kernel=g.KERNEL_RING)
        g.imdp_session_run(sess)
        want = np.zeros(small.n_states)
        g.imdp_session_read(sess, 0, want)
        sess.close()
        np.testing.assert_array_equal(V, want)
    # the others are far from their ends (1.3 s each alone)
    assert [g.imdp_server_poll(server, t) for t in slows + [long]] == [g.IMDP_EPENDING] * 4
    assert g.imdp_server_launches(server)["per_iteration"] == 0
    server.close()
    mw.close()
    ms.close()
