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
