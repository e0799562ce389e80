"""bench.py's stored ncu counters of the warp sweep belong to the capture that profiles/
summarises and to the sources as they are, and are reported for that configuration only."""
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

CASE = dict(storage="f32", workload="channel_4096x512", physics="full", cols_per_thread=2)


def test_counters_match_the_profile_summary():
    text = open(os.path.join(ROOT, "profiles", "k_sweep_channel_4096x512.md")).read()
    assert f"`{bench.SWEEP_COUNTERS_SOURCE}`" in text
    m = re.search(r"dram__bytes_write\.sum \| ([\d.]+) \+ ([\d.]+) = ", text)
    mb = float(m.group(1)) + float(m.group(2))
    assert abs(bench.SWEEP_F32_4096x512_DRAM_BYTES / 1e6 - mb) < 0.011
    m = re.search(r"warp instructions executed \| ([\d.]+) M", text)
    assert abs(bench.SWEEP_F32_4096x512_WARP_INSTR / 1e6 - float(m.group(1))) < 0.006


def test_the_default_run_has_counters():
    dram, instr, built, captured = bench.stored_counters("k_sweep", **CASE)
    assert built == captured
    assert dram == bench.SWEEP_F32_4096x512_DRAM_BYTES
    assert instr == bench.SWEEP_F32_4096x512_WARP_INSTR


def test_no_counters_for_other_runs(monkeypatch):
    for other in (dict(storage="f16"), dict(workload="channel_1024x128"), dict(physics="none")):
        assert bench.stored_counters("k_sweep", **{**CASE, **other})[:2] == (None, None)
    assert bench.stored_counters("k_tile", **CASE)[:2] == (None, None)
    assert bench.stored_counters("k_fused_step", **CASE)[:2] == (None, None)  # two columns
    monkeypatch.setattr(bench, "SWEEP_COUNTERS_SOURCE", "0")  # sources changed since
    assert bench.stored_counters("k_sweep", **CASE)[:2] == (None, None)
