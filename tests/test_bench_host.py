"""Host-side parts of bench.py without a GPU: the clock record that decides whether a
run is kept, the roofline peak, and the rule that profiled DRAM traffic is reported only
for the kernel sources it was captured on."""
import json
import os

import bench


def _sample(sm, mx, hw="Not Active", hwt="Not Active", swt="Not Active", cap="Not Active"):
    return ["0", str(sm), str(mx), "900.0", hw, hwt, swt, cap]


def test_clock_summary_takes_the_median_and_collects_active_reasons():
    c = bench.ClockSampler()
    c.samples = [_sample(2070, 2070), _sample(1980, 2070, cap="Active"), _sample(2070, 2070),
                 _sample(1500, 2070, hwt="Active")]
    s = c.summary()
    assert s["sm_mhz"] == 2025.0 and s["sm_max_mhz"] == 2070.0 and s["samples"] == 4
    assert s["reasons"] == ["hw_thermal_slowdown", "sw_power_cap"]


def test_clock_summary_without_samples_says_so():
    s = bench.ClockSampler().summary()
    assert s["sm_mhz"] is None and s["reasons"] == ["unsampled"]


def test_peak_is_the_measured_copy_bandwidth_else_the_fallback():
    peak, kind = bench._peaks()
    path = os.path.join(bench.ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as fh:
            assert kind == "measured" and peak == float(json.load(fh)["hbm_gbs"])
    else:
        assert (peak, kind) == (6800.0, "fallback")


def test_profiled_traffic_only_for_the_sources_it_was_captured_on(monkeypatch):
    with open(os.path.join(bench.ROOT, "profiles", "traffic.json")) as fh:
        d = json.load(fh)
    key = "rb_4096x2048_fp32"
    monkeypatch.setattr(bench, "_kernel_source_hash", lambda: d[key]["source_hash"])
    assert bench._profiled_traffic(key) == d[key]["read"] + d[key]["write"] == d[key]["bytes_per_launch"]
    monkeypatch.setattr(bench, "_kernel_source_hash", lambda: "0" * 16)
    assert bench._profiled_traffic(key) is None
    assert bench._profiled_traffic("no_such_workload") is None


def test_profiled_traffic_sees_the_resident_kernel_and_the_steps_of_a_launch(monkeypatch, tmp_path):
    # an edit of any step kernel's source withdraws the record, and the bytes of a launch of one
    # number of steps are not those of another
    real = bench._kernel_source_hash()
    for rel in ("tclbm_device.cuh", "tclbm_tma.cuh", "tclbm_resident.cuh"):
        assert any(s.endswith(rel) for s in bench.KERNEL_SOURCES)
    for k in range(len(bench.KERNEL_SOURCES)):
        monkeypatch.setattr(bench, "KERNEL_SOURCES", bench.KERNEL_SOURCES[:k] + bench.KERNEL_SOURCES[k + 1:])
        assert bench._kernel_source_hash() != real
        monkeypatch.undo()
    (tmp_path / "profiles").mkdir()
    rec = {"w": {"bytes_per_launch": 7, "source_hash": real, "steps_per_launch": 64}}
    (tmp_path / "profiles" / "traffic.json").write_text(json.dumps(rec))
    monkeypatch.setattr(bench, "_kernel_source_hash", lambda: real)
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert bench._profiled_traffic("w", 64) == 7
    assert bench._profiled_traffic("w", 1000) is None and bench._profiled_traffic("w") is None


def test_launches_of_a_call():
    desc = "tclbm_step_tile<32,4,float> grid (8, 32) block (128); 12 steps or more: tclbm_resident grid (19, 8) block (288)"
    assert [bench._step_launches(desc, n) for n in (11, 12, 1000, 1024, 1030, 2048, 3000)] == [11, 1, 1, 1, 7, 2, 3]
    assert bench._step_launches("tclbm_step_tma_corr<128,float> grid (32, 32)", 70) == 70
