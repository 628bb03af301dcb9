"""Little device memory left: what the per-iteration kernels and one-by-one reads
can do in it is done. The GPU's memory is taken by tensors; every kernel has run
before, so nothing is loaded meanwhile. Each case has a process of its own, since the
memory that a process's pool keeps is given back when an allocation needs it."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import paper_2401_04068_gb300 as g
from workloads import banded_imdp

pytestmark = pytest.mark.gpu
MB = 1 << 20


class Leave:
    """Takes device memory until about ``free`` bytes are left."""

    def __init__(self, free):
        self.free = free

    def __enter__(self):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.held = []
        for _ in range(4):
            take = (torch.cuda.mem_get_info()[0] - self.free) // (2 * MB) * (2 * MB)
            if take < 10 * MB:  # (smaller tensors share blocks of 20 MB)
                break
            try:
                self.held.append(torch.empty(take, dtype=torch.uint8, device="cuda"))
            except torch.OutOfMemoryError:
                self.held.append(torch.empty(take - 64 * MB, dtype=torch.uint8, device="cuda"))
        return self

    def __exit__(self, *a):
        self.held.clear()
        torch.cuda.empty_cache()


def session_without_room_for_its_plan():
    # the grid kernel's lists of missed columns (64 B a column) do not fit
    m = banded_imdp(200000, 2, 200000 * 2 * 6 + 1, eps=0.1, seed=1)
    model = g.create_model(m)
    spec = g.make_spec(horizon=12, reach=m.goal)

    def run(kernel=g.KERNEL_RULE):
        sess = g.imdp_session_create([model], [spec])
        g.imdp_session_set_launch(sess, kernel=kernel)
        route = g.imdp_session_step_route(sess, 12)["kernel"]
        g.imdp_session_run(sess)
        raw, k = g.imdp_session_checkpoint(sess, 0)
        sess.close()
        return route, raw, k

    _, ref, _ = run(g.KERNEL_RING)
    assert run()[0] == g.KERNEL_GRID
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    sess = g.imdp_session_create([model], [spec])
    need = free - torch.cuda.mem_get_info()[0]
    sess.close()
    assert need >= 30 * MB
    with Leave(need - 16 * MB):
        assert torch.cuda.mem_get_info()[0] < need - 5 * MB
        route, raw, k = run()
    assert route not in (g.KERNEL_GRID, g.KERNEL_RESIDENT) and k == 12
    np.testing.assert_array_equal(raw, ref)
    model.close()


def batch_results_without_room_for_all_of_them():
    # 32 models of a million absorbing states: their results are 256 MB together, 8 MB each
    n = 1000000
    ptr = np.arange(n + 1, dtype=np.int32)
    one = np.ones(n)
    model = g.imdp_create_csc(n, n, n, ptr, ptr, ptr[:n], one, one)
    count = 32
    specs = [g.make_spec(horizon=2 + i % 3, reach=np.arange(i, n, 7, dtype=np.int32)) for i in range(count)]
    outs = [np.full(n, -1.0) for _ in range(count)]
    g.imdp_value_iteration_batch([model] * count, specs, outs, [0] * count)
    want = [o.copy() for o in outs]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    sess = g.imdp_session_create([model] * count, specs)
    need = free - torch.cuda.mem_get_info()[0]
    sess.close()
    for o in outs:
        o[:] = -1.0
    ks = [0] * count
    with Leave(need + 24 * MB):
        assert torch.cuda.mem_get_info()[0] < need + 36 * MB
        assert g.imdp_value_iteration_batch([model] * count, specs, outs, ks) == g.IMDP_OK
    assert ks == [2 + i % 3 for i in range(count)]
    for i, (o, w) in enumerate(zip(outs, want)):
        np.testing.assert_array_equal(o, w)
        np.testing.assert_array_equal(o, (np.arange(n) % 7 == i % 7) & (np.arange(n) >= i))
    model.close()


def plan_change_without_room():
    # one tile a state: a table of 36 MB, which does not fit; steps then report that
    # there is no plan (the old one's memory is gone) until one is set
    n = 1000000
    ptr = np.arange(n + 1, dtype=np.int32)
    one = np.ones(n)
    model = g.imdp_create_csc(n, n, n, ptr, ptr, ptr[:n], one, one)
    spec = g.make_spec(horizon=9, reach=np.arange(0, n, 3, dtype=np.int32))
    sess = g.imdp_session_create([model], [spec])
    g.imdp_session_set_launch(sess, kernel=g.KERNEL_RING)
    g.imdp_session_step(sess, 3)
    with Leave(12 * MB):
        with pytest.raises(g.ImdpError) as e:
            g.imdp_session_set_launch(sess, kernel=g.KERNEL_RING, tile_entries=1)
        assert e.value.status == g.IMDP_ENOMEM
        with pytest.raises(g.ImdpError) as e:
            g.imdp_session_step(sess, 1)
        assert e.value.status == g.IMDP_ENOMEM
    g.imdp_session_set_launch(sess, kernel=g.KERNEL_RING)
    g.imdp_session_run(sess)
    V, k = np.zeros(n), [0]
    assert g.imdp_session_read(sess, 0, V, k) == g.IMDP_OK and k[0] == 9
    np.testing.assert_array_equal(V, np.arange(n) % 3 == 0)
    sess.close()
    model.close()


@pytest.mark.parametrize("case", ["session_without_room_for_its_plan", "batch_results_without_room_for_all_of_them",
                                  "plan_change_without_room"])
def test_little_memory(case):
    here = os.path.dirname(os.path.abspath(__file__))
    torch.cuda.empty_cache()
    code = f"import sys; sys.path[:0] = [{os.path.dirname(here)!r}, {here!r}]; import test_memory_gpu as t; t.{case}()"
    out = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
