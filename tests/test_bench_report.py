"""What the benchmark's line says of the joint fit."""


def test_fit_time_is_that_of_a_step_and_all_its_launches():
    import bench
    r = bench.fit_report((1.95, 70), 10, 96)           # ten steps of seven launches, 0.195 ms per step
    assert r["launches_per_step"] == 7 and abs(r["ms"] - 0.195) < 1e-12 and r["groups"] == 96
    assert bench.fit_report(None, 10, 96)["ms"] is None
