"""The measured traffic of bench.py belongs to launches that the bench makes, and reaches its roofline record."""
import bench
import workloads as W


def test_traffic_reaches_the_roofline_record():
    by_name = {f().name: f() for f in W.ALL.values()}
    assert len(bench.TRAFFIC) == 4
    for (name, cat, rows), t in bench.TRAFFIC.items():
        w = by_name[name]
        assert rows % w.n == 0 and 1 <= rows // w.n <= w.k
        rec = bench.kernel_model(cat, w, "fp32", 100, 10, 1000.0, rows, "path=cuda-core 2-D step kernel")
        assert rec["traffic"] == t["bytes"] * 100 and rec["traffic_src"] == t["src"]
        assert bench.kernel_model(cat, w, "bf16", 100, 10, 1000.0, rows, "path=x")["traffic"] is None


def test_mean_steps_per_launch():
    """3-D workload, two marches in groups of two vectors with tiles of 512: 10 whole tiles and one of 20 steps."""
    w = next(f() for f in W.ALL.values() if f().name.startswith("adv3d"))
    n_t = 1285
    assert bench.steps_per_launch("march", w, n_t, 2, 2 * 4 * 11, 2) == 2 * 4 * 5140 / 88
    assert bench.steps_per_launch("analysis", w, n_t, 2, 32, 2) == 2 * 4 * n_t / 32
    d = next(f() for f in W.ALL.values() if f().name.startswith("dense"))
    assert bench.steps_per_launch("synthesis", d, 400, 1, 2, d.k) == 200
