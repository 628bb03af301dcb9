"""The bench line names the kernel that ran, its launches, and what bounds it."""
import bench


def _launch(kernel, copied=0):
    return {"chosen_by": "rule", "kernel": 2, "route": {"kernel": kernel, "launches": 1, "copied": copied}}


def test_kernel_names_follow_the_route():
    names = [bench.kernel_name(_launch(k)) for k in range(1, 7)]
    assert names == ["bellman_step_kernel", "bellman_direct_kernel", "bellman_tiny_kernel", "bellman_slice_kernel",
                     "bellman_cluster_kernel", "bellman_grid_kernel"]


def test_roofline_charges_memory_with_what_comes_from_it():
    # 200 iterations of a 2 GB model in 60 ms: per iteration it streams from HBM; a
    # kernel that keeps it on chip reads it once a launch
    args = (200 * 2e9, 2e9, 2e9, 0.06, 6800.0)
    for kernel in (1, 2, 4):
        r = bench.roofline(_launch(kernel), *args)
        assert r["bound"] == "hbm" and abs(r["achieved"] - 6666.67) < 0.01 and r["frac"] == r["achieved"] / 6800.0
    r = bench.roofline(_launch(5), *args)
    assert "L2" in r["bound"] and abs(r["achieved"] - 33.33) < 0.01 and abs(r["on_chip_gbs"] - 6666.67) < 0.01
    assert "shared memory" in bench.roofline(_launch(5, 1), *args)["bound"]
    # the grid kernel streams a model that L2 does not hold, and reads a smaller one from L2
    assert bench.roofline(_launch(6), *args)["bound"] == "hbm"
    small = (200 * 1e8, 1e8, 1e8, 0.06, 6800.0)
    assert "L2" in bench.roofline(_launch(6), *small)["bound"]
    assert "shared memory" in bench.roofline(_launch(6, 1), *small)["bound"]
