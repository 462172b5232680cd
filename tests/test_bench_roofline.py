"""The bench line's closure rates are what the kernels executed and read (committed captures
over live times), never the work of a list walk that bit rows replaced."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CS = {"probes": 4_000_000_000, "gathers": 10_000_000, "out_entries": 40_000_000}
TIMES = {"close_bits256": [6.0, 2], "close_bits128": [4.0, 2], "close_bucket": [0.1, 2],
         "wedge_gather": [2.2, 2]}   # summed ms and launches of 2 steps


def roofline(tmp_path, monkeypatch, entries):
    if ROOT not in sys.path:
        sys.path.insert(0, ROOT)
    import bench

    csrc = tmp_path / "paper_2504_02271_gb300" / "csrc"
    csrc.mkdir(parents=True)
    (csrc / "k.cu").write_text("kernel\n")
    (tmp_path / "profiles").mkdir()
    sha = bench.source_sha(str(csrc / "k.cu"))
    d = {n: {"source": "k.cu", "source_sha": sha if ok else "stale", "dram_bytes_per_launch": b,
             "inst_executed_per_launch": i} for n, (b, i, ok) in entries.items()}
    (tmp_path / "profiles" / "dram_traffic.json").write_text(json.dumps(d))
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    return bench.closure_roofline(TIMES, CS, 10**9, {"sm_mhz": 2000.0}, 2, "w")


def test_rates_come_from_the_captures(tmp_path, monkeypatch):
    r = roofline(tmp_path, monkeypatch, {"close_bits256/w": (3e8, 2.0e9, True),
                                         "close_bits128/w": (2e8, 1.5e9, True)})
    # 5 ms of captured kernels per step: 3.5e9 warp instructions, 0.5 GB
    assert abs(r["achieved"] - 0.7) < 1e-9 and r["unit"] == "T warp instructions/s"
    assert r["frac"] == round(0.7 / (152 * 4 * 2000.0e6 / 1e12), 4)
    assert r["hbm"]["achieved"] == 100.0 and r["traffic"] == 500_000_000
    assert r["covers"] == 1.0


def test_kernels_without_a_current_capture_are_left_out(tmp_path, monkeypatch):
    r = roofline(tmp_path, monkeypatch, {"close_bits256/w": (3e8, 2.0e9, True),
                                         "close_bits128/w": (2e8, 1.5e9, False)})
    assert r["covers"] == 0.6 and r["hbm"]["achieved"] == 100.0
    assert abs(r["achieved"] - 2.0e9 / 3e-3 / 1e12) < 1e-4


def test_no_capture_no_rate(tmp_path, monkeypatch):
    r = roofline(tmp_path, monkeypatch, {})
    assert r["achieved"] is None and r["frac"] is None and r["covers"] == 0.0
    assert r["hbm"]["achieved"] is None and r["hbm"]["frac"] is None and r["traffic"] is None
    # the list walk's work is printed for comparison, without a rate or a fraction
    assert r["list_walk"]["bytes"] == 4 * CS["probes"] + 20 * CS["out_entries"] + 4 * CS["gathers"]
    assert not {"frac", "achieved", "peak"} & set(r["list_walk"])
