"""States of very many actions: a model's creation spreads their columns over the
GPU, and what it finds out about their destinations (parts, windows) is right."""
import time

import numpy as np
import pytest

import paper_2401_04068_gb300 as g
from test_resident_gpu import _run, _same
from workloads import banded_imdp
from workloads.imdp_synth import IMDPInput, concat_block_diagonal

pytestmark = pytest.mark.gpu


def _actions(n, counts, k=6, seed=3):
    """`counts[s]` actions of state s (2 where not given), k scattered destinations each."""
    rng = np.random.default_rng(seed)
    a = np.full(n, 2)
    for s, c in counts.items():
        a[s] = c
    cols = int(a.sum())
    k = min(k, n)
    strip = n // k
    rows = rng.integers(0, strip, (cols, k)) + np.arange(k) * strip  # ascending: one in each strip
    p = rng.random((cols, k)) + 0.05
    p /= p.sum(1, keepdims=True)
    return IMDPInput(n, np.concatenate([[0], np.cumsum(a)]).astype(np.int32),
                     (np.arange(cols + 1) * k).astype(np.int32), rows.ravel().astype(np.int32),
                     (p * (1 - 0.2 * rng.random(p.shape))).ravel(), np.minimum(1, p * (1 + 0.2 * rng.random(p.shape))).ravel(),
                     np.arange(2, dtype=np.int32))


def test_creation_does_not_wait_for_one_thread():
    m = _actions(200, {100: 100000})
    best = 1.0
    for _ in range(5):
        t = time.perf_counter()
        g.create_model(m).close()
        best = min(best, time.perf_counter() - t)
    assert best < 0.006, best  # 20 ms when one thread goes through the state's columns, 1 without that


# around the length from which a state's columns are spread, and states of a warp's and a block's columns
@pytest.mark.parametrize("counts", [{3: 33}, {0: 31, 1: 32, 2: 33, 3: 64, 50: 65}, {10: 600, 11: 1, 12: 300}])
def test_parts_and_windows_of_long_states(counts):
    long = _actions(60, counts)
    near = banded_imdp(3000, 1, 3000 * 81 + 1, eps=0.1, seed=5)
    for m, kernel in ((long, None), (concat_block_diagonal([long, near]), g.KERNEL_GRID),
                      (concat_block_diagonal([long] * 40), g.KERNEL_RESIDENT)):
        model = g.create_model(m)
        specs = [g.make_spec(horizon=15, reach=m.goal)]
        if kernel:
            sess = g.imdp_session_create([model], specs)
            assert g.imdp_session_step_route(sess, 15)["kernel"] == kernel
            sess.close()
        _same(_run([model], [m], specs, g.KERNEL_RING, policy=True), _run([model], [m], specs, g.KERNEL_RULE, policy=True))
        model.close()
