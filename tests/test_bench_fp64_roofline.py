"""The FP64 arm's roofline counts what the kernel gives the FP64 pipe: its own
time of a trajectory (2^20 sites, 100 steps: 1.48 ms) cannot exceed the pipe's
measured rate, 0.62e12 FMA/s."""


def test_fraction_is_a_fraction():
    import bench
    r = bench.fp64_roofline(1.48e-3, 0.62e12)
    assert r["ops_per_site_step"] == 7
    assert abs(r["achieved"] - 7 * 2 ** 20 * 100 / 1.48e-3 / 1e12) < 1e-9
    assert 0.7 < r["frac"] < 1.0
