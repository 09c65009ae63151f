"""When a captured traffic figure counts in bench.py's roofline line."""
import bench
from tests.test_bench_host import _fake


def test_traffic_belongs_to_the_launch_per_class_kernels(monkeypatch):
    info, s, peaks, n, ms = _fake()
    monkeypatch.setattr(bench, "kernel_source_hash", lambda: "h0")
    monkeypatch.setattr(bench, "TRAFFIC", {("refresh", "mixed", "h0"): 5.0e6, ("solve", "mixed", "h0"): 1.0e6})
    for kind in ("refresh", "solve"):
        assert bench.roofline(info, s, kind, "mixed", ms, n, peaks)["traffic"] > 0
        assert bench.roofline(info, s, kind, "mixed", ms, n, peaks, by_class=False)["traffic"] is None


def test_hash_follows_the_sources_that_the_figure_is_of(monkeypatch, tmp_path):
    csrc = tmp_path / "paper_2312_04998_gb300" / "csrc"
    csrc.mkdir(parents=True)
    for name in ("integrate.cu", "integ.h", "kern_rhs.cu", "cell.cu"):
        (csrc / name).write_text("int a;  // one\n")
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    h = bench.kernel_source_hash()
    for name, same in (("cell.cu", True), ("integrate.cu", False), ("integ.h", False), ("kern_rhs.cu", False)):
        (csrc / name).write_text("int b;\n")
        assert (bench.kernel_source_hash() == h) is same, name
        (csrc / name).write_text("int a;\n/* another comment */\n")
        assert bench.kernel_source_hash() == h
