"""A session's device memory: many plan changes neither free memory in use nor
grow without bound (on the CPU, with watched host memory; and with real plans)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_buffers_stay_apart_over_many_plan_changes(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "buffers_client")
    subprocess.run([cxx, "-std=c++17", "-Wall", "-Wextra", "-Werror", "-O1", "-g", "-I",
                    os.path.join(ROOT, "paper_2401_04068_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "buffers_client.cpp"), "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(5000, 1, 39), (20000, 2, 19)])
def test_many_plans_in_one_session(shape):
    import paper_2401_04068_gb300 as g
    from workloads import banded_imdp
    n, a, k = shape
    m = banded_imdp(n, a, n * a * (k + 1) + 1, eps=0.1, seed=n)
    model = g.create_model(m)
    spec = g.make_spec(horizon=150, reach=m.goal)
    cfgs = [dict(kernel=g.KERNEL_RING, tile_entries=3072), dict(kernel=g.KERNEL_DIRECT, tile_entries=1024),
            dict(kernel=g.KERNEL_RING, tile_entries=500), dict(kernel=g.KERNEL_SLICE)]
    words = []
    for plans in (1, 100):
        sess = g.imdp_session_create([model], [spec])
        for i in range(100):
            if i < plans:
                g.imdp_session_set_launch(sess, **cfgs[i % len(cfgs)])
            g.imdp_session_step(sess, 1)
        words.append(g.imdp_session_checkpoint(sess, 0))
        sess.close()
    assert words[0][1] == words[1][1] == 100
    np.testing.assert_array_equal(words[0][0], words[1][0])
    model.close()
