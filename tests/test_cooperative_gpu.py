"""The grid kernel's cooperative launch when it cannot be had, and its bounded wait
when it runs out (both by test hooks on the host; no GPU fault is involved)."""
import time

import numpy as np
import pytest
import torch

import paper_2401_04068_gb300 as g
from workloads import banded_imdp

pytestmark = pytest.mark.gpu


def _case():
    m = banded_imdp(2500, 1, 2500 * 120 + 2500 + 1, eps=0.1, seed=41)
    return m, g.create_model(m)


def _ring(model, spec):
    sess = g.imdp_session_create([model], [spec])
    g.imdp_session_set_launch(sess, kernel=g.KERNEL_RING)
    g.imdp_session_run(sess)
    out = g.imdp_session_checkpoint(sess, 0)
    sess.close()
    return out


@pytest.mark.parametrize("stream", [False, True])
def test_sessions_go_on_per_iteration(stream):
    m, model = _case()
    spec = g.make_spec(horizon=40, reach=m.goal)
    ref, _ = _ring(model, spec)
    st = torch.cuda.Stream() if stream else None
    sess = g.imdp_session_create([model], [spec], stream=st)
    assert g.imdp_session_step_route(sess, 20)["kernel"] == g.KERNEL_GRID
    g.imdp_session_step(sess, 7, st)
    g.imdp_debug_refuse_cooperative(True)
    try:
        g.imdp_session_step(sess, 20, st)
    finally:
        g.imdp_debug_refuse_cooperative(False)
    assert g.imdp_session_launches(sess) == 27
    assert g.imdp_session_step_route(sess, 20)["kernel"] not in (g.KERNEL_GRID, g.KERNEL_RESIDENT)
    g.imdp_session_run(sess, stream=st)
    raw, k = g.imdp_session_checkpoint(sess, 0, stream=st)
    assert k == 40
    np.testing.assert_array_equal(raw, ref)
    sess.close()
    model.close()


def test_servers_go_on_per_iteration():
    m, model = _case()
    spec = g.make_spec(horizon=40, reach=m.goal)
    ref, _ = _ring(model, spec)
    server = g.imdp_server_create(64 << 20)
    g.imdp_debug_refuse_cooperative(True)
    try:
        tickets = [g.imdp_server_submit(server, model, spec) for _ in range(5)]
        for t in tickets:
            V, k = np.zeros(m.n_states), [0]
            assert g.imdp_server_wait(server, t, 60000.0, V, k) == g.IMDP_OK and k[0] == 40
            np.testing.assert_array_equal(V, ref.astype(np.float64) / 2.0 ** 63)
        time.sleep(0.2)
        n = g.imdp_server_launches(server)
        assert n["shared"] == 0 and n["per_iteration"] > 0
    finally:
        g.imdp_debug_refuse_cooperative(False)
    server.close()
    model.close()


def test_bounded_grid_barrier_reports_timeout_and_context_survives():
    m, model = _case()
    spec = g.make_spec(horizon=40, reach=m.goal)
    ref, _ = _ring(model, spec)
    sess = g.imdp_session_create([model], [spec])
    assert g.imdp_session_step_route(sess, 20)["kernel"] == g.KERNEL_GRID
    V = np.zeros(m.n_states)
    g.imdp_debug_stall_producer(True)
    try:
        t = time.time()
        g.imdp_session_step(sess, 20)
        st = g.imdp_session_read(sess, 0, V, check=False)
        elapsed = time.time() - t
    finally:
        g.imdp_debug_stall_producer(False)
    assert st == g.IMDP_ETIMEOUT
    assert elapsed < 30.0  # bounded: the waits gave up on their own
    assert not V.any()  # no output of a failed run
    # the same session, reset, runs normally afterwards
    g.imdp_session_reset(sess)
    g.imdp_session_step(sess, 40)
    raw, k = g.imdp_session_checkpoint(sess, 0)
    assert k == 40
    np.testing.assert_array_equal(raw, ref)
    sess.close()
    model.close()
