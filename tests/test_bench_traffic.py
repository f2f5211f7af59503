"""bench.py reports captured DRAM traffic only for the sources that were
captured (no GPU)."""
import bench
from paper_2303_18244_gb300.generator import recursion


def test_digest_follows_the_generated_code(monkeypatch):
    own = bench.kernel_digest("ggttgg")
    assert own == bench.kernel_digest("ggttgg")
    text = recursion.emit_recursion(4, "ggttgg")
    monkeypatch.setattr(recursion, "emit_recursion", lambda n, tag: text.replace("R(0.25)", "R(0.250)"))
    assert bench.kernel_digest("ggttgg") != own


def test_traffic_counts_the_results_and_needs_the_captured_sources(monkeypatch):
    monkeypatch.setattr(bench, "NCU_TRAFFIC", {"ggttgg": (1000, 200000, bench.kernel_digest("ggttgg"))})
    assert bench.traffic_per_launch("ggttgg", 3000) == 3 * 200000 + 8 * 3000
    monkeypatch.setattr(bench, "NCU_TRAFFIC", {"ggttgg": (1000, 200000, "0" * 16)})
    assert bench.traffic_per_launch("ggttgg", 3000) is None
    assert bench.traffic_per_launch("eemumu", 3000) is None
