"""Little device memory left: what the per-iteration kernels and one-by-one reads
can do in it is done. The GPU's memory is taken by tensors; every kernel has run
before, so nothing is loaded meanwhile."""
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


def test_a_session_without_room_for_its_plan():
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


def test_batch_results_without_room_for_all_of_them():
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
