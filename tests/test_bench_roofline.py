"""bench.py's roofline counts what the kernel executes: its warp instructions
against the rate at which they can issue."""
import bench


def test_issue_roofline(monkeypatch):
    monkeypatch.setattr(bench, "measured", lambda workload, what: {"warp_instructions": 10 ** 8, "bytes": 5}[what])
    r = bench.issue_roofline("stress", ms=0.2, sms=100, mhz=2000.0, mixed_per_s=25.6e12)
    assert r["peak"] == 0.8 and r["achieved"] == 0.5 and r["frac"] == 0.625   # 400 a clock; 10^8 in 0.2 ms
    assert r["peak_measured"] == 0.8 and r["traffic"] == 5


def test_no_figure_without_a_count_of_these_sources(monkeypatch):
    monkeypatch.setattr(bench, "measured", lambda workload, what: None)
    r = bench.issue_roofline("stress", ms=0.2, sms=100, mhz=2000.0, mixed_per_s=25.6e12)
    assert r["achieved"] is None and r["frac"] is None


def test_committed_records_count_instructions():
    assert all(r["warp_instructions"] > 0 for r in bench.NCU_TRAFFIC.values())
