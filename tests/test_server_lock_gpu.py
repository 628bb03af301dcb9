"""Callers of the server are not held up while it plans, and a mix of requests that
does not fit the grid kernel together is not planned over and over."""
import threading
import time

import numpy as np
import pytest

import paper_2401_04068_gb300 as g
from workloads import banded_imdp

pytestmark = pytest.mark.gpu


def test_callers_do_not_wait_for_a_plan():
    # each of these needs 90 CTAs and more: no two fit together
    ms = [banded_imdp(150000, 2, 150000 * 2 * 6 + 1, eps=0.1, seed=100 + i) for i in range(3)]
    models = [g.create_model(m) for m in ms]

    def burst():
        server = g.imdp_server_create(1 << 30)
        waits, stop = [0.0], False

        def caller():
            while not stop:
                t = time.perf_counter()
                g.imdp_server_stats(server)
                waits.append(time.perf_counter() - t)
                time.sleep(2e-4)

        thread = threading.Thread(target=caller)
        thread.start()
        tickets = []
        for i in range(12):
            tickets.append(g.imdp_server_submit(server, models[i % 3], g.make_spec(horizon=100, reach=ms[i % 3].goal)))
            time.sleep(0.002)
        outs = [np.zeros(150001) for _ in tickets]
        for t, V in zip(tickets, outs):
            assert g.imdp_server_wait(server, t, 120000.0, V) == g.IMDP_OK
        stop = True
        thread.join()
        time.sleep(0.1)
        s = g.imdp_server_stats(server)
        server.close()
        return max(waits), s["wall_ms"] - s["device_ms"], outs

    worst, host_ms = 1.0, 1e9
    for _ in range(3):
        w, h, outs = burst()
        worst, host_ms = min(worst, w), min(host_ms, h)
    # 17 ms under the mutex, and 45 ms of the worker's time beside the GPU's
    assert worst < 0.008, worst
    assert host_ms < 25.0, host_ms
    for i in range(3):
        sess = g.imdp_session_create([models[i]], [g.make_spec(horizon=100, reach=ms[i].goal)])
        g.imdp_session_set_launch(sess, kernel=g.KERNEL_RING)
        g.imdp_session_run(sess)
        V = np.zeros(150001)
        g.imdp_session_read(sess, 0, V)
        sess.close()
        for o in outs[i::3]:
            np.testing.assert_array_equal(o, V)
        models[i].close()


def test_no_cuts_for_a_plan_that_has_no_room():
    # the budget holds the requests and little more; the lists of missed columns (64 B
    # a column) find no room, which the worker sees without cutting the models
    n, count = 45000, 10
    ms = [banded_imdp(n, 1, n * 7 + 1, eps=0.1, seed=200 + i) for i in range(count)]
    models = [g.create_model(m) for m in ms]
    host_ms = 1e9
    for _ in range(3):
        server = g.imdp_server_create(count * (37 * (n + 1)) + (1 << 20))
        tickets = [g.imdp_server_submit(server, x, g.make_spec(horizon=40 + 16 * i, reach=m.goal))
                   for i, (x, m) in enumerate(zip(models, ms))]
        for t in tickets:
            assert g.imdp_server_wait(server, t, 120000.0, np.zeros(n + 1)) == g.IMDP_OK
        time.sleep(0.1)
        s, launches = g.imdp_server_stats(server), g.imdp_server_launches(server)
        host_ms = min(host_ms, s["wall_ms"] - s["device_ms"])
        server.close()
    assert launches["per_iteration"] > 0
    assert host_ms < 6.5, host_ms  # 3.0; 8.0 when it cuts them
    for x in models:
        x.close()
