"""The bench's work model of the row build's analysis: the flops of its sums, counted one by one."""
import bench
import inputs


def test_analysis_flops_are_those_of_the_sums():
    for p in (1, 4, 17):
        lat, N = 2 * p + 2, 4 * p + 4
        fourier = sum(2 * N + sum(2 * (N // 4) for _ in range(2 * p + 1)) for _ in range(lat))
        legendre = sum(2 * lat * 2 for m in range(p + 1) for n in range(m, p + 1))
        assert bench.analysis_flops_per_target(p) == 14 * (fourier + legendre)


def test_roofline_of_the_analysis():
    cfg = inputs.config3(seed=3)
    ms = {"self_analysis": 500.0, "pairs_fp32": 100.0}
    r = bench.roofline(ms, {"self_analysis": 392, "pairs_fp32": 20}, {"pairs_fp32": 1e12}, cfg, {"ffma": {"value": 80.0}})
    work = 2 * sum((d.p + 1) * (2 * d.p + 2) * bench.analysis_flops_per_target(d.p) for d in cfg.drops)
    assert r["kernel_class"] == "self_analysis" and abs(r["achieved"] - work / 0.5 / 1e12) < 1e-9
    assert abs(r["frac"] - r["achieved"] / 80.0) < 1e-12
