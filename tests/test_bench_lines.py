"""The bench line's bounds name what the kernel can meet (CPU)."""
import bench
from paper_2212_04551_gb300 import graphs as G


def test_no_l2_bound_where_the_marks_are_in_shared_memory(monkeypatch):
    monkeypatch.setattr(bench, "l2_peaks", lambda: {"stream_gbs": 2.0, "sector_gbs": 1.0})
    arm = {"kernel_ms": 1.0, "adjacency_entries": 10 ** 9}
    small = bench.motif_roofline(arm, G.sbm(2000, 100, 0.5, 0.01, 4), 6)
    assert small["bound"] != "l2" and small["frac"] is None and small["achieved"] == 1000.0
    large = bench.motif_roofline(arm, G.erdos_renyi_m(40000, 50000, 1), 5)
    assert large["bound"] == "l2" and large["frac"] == large["achieved"] / large["peak"]


def test_marks_of_twelve_kilobytes():
    """n marks (to a multiple of 16) and the arrays of levels 1 .. k - 2."""
    path = G.path(12288 - 16 - 4 * 20)                  # k = 4, degree 2: 8 + 8 ints to 20 x 4 bytes at most
    assert bench.marks_in_shared(path, 4)
    assert not bench.marks_in_shared(G.path(12288), 4)
