"""The bench's printed line: short enough for a record that keeps the last 3,000 characters of
its output, with every key of the measured workload."""

import json

import pytest

pytest.importorskip("torch")

import bench  # noqa: E402

NOTE = "x" * 400


def _record():
    """A full run's record, floats at full length."""
    f = 0.12345678901234567
    point = {"spikers": 0, "events": 1e8 * f, "ms": f, "events_per_s": 1e12 * f, "bytes": 1e9 * f, "gbs": 1e4 * f,
             "frac": f, "ring_entries_updated": 1e7 * f, "speedup_vs_plain": f}
    points = [dict(point, spikers=s, order=o) for s in (2048, 8192, 20480) for o in ("random", "sorted")]
    plain = [dict(point, spikers=s) for s in (2048, 8192, 20480)]
    return {
        "metric": bench.METRIC, "value": 34351234567.123456, "unit": "synaptic events/s", "n_gpus": 8, "steps": 20,
        "warmup": 5, "ms_per_step": 2.9890123456789, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32/i32", "data": "synthetic (PD microcircuit sampled from the paper's tables)",
        "config": {"workload": "pd_full: 77,169 neurons, 284,811,022 synapses, dt 0.1 ms, seed 1+rank",
                   "ticks_per_step": 1024, "bio_seconds": 2.048, "steps_per_graph": 1024, "engine": "pipelined",
                   "deliver_blocks": 304, "parallelism": "replicas x8", "l2": NOTE[:100]},
        "rtf": f, "realtime_x": 34.123456789012345, "spikes_per_tick": 28.43208, "events_per_tick": 100268.87094726562,
        "instances": {"n": 10, "steps_each": 10240, "rtf_mean": f, "rtf_sd": f, "instances": [{"rtf": f}] * 10, "note": NOTE},
        "events_incl_thalamic": {"value": 1e11 * f, "note": NOTE},
        "e2e": {"value": 3.4e10 + f, "unit": "synaptic events/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 232949.2,
                "note": NOTE},
        "gpu_launches": 20500,
        "roofline": {"kernel": "k_step", "bound": "hbm", "achieved": 1e4 * f, "peak": 6781.1, "unit": "GB/s", "frac": f,
                     "traffic": 1161472, "peak_source": "measured hbm_gbs (copy bandwidth, burst)"},
        "kernels": {"k_step": {"avg_us": 2.9 + f, "gbs": 1e4 * f, "note": NOTE}},
        "compressed_records": {k: {"rtf": f, "delivery_saturating": plain, "note": NOTE}
                               for k in ("int8_pair", "bf16", "blocked6", "blocked4", "blocked8")},
        "workloads": {k: {"us_per_step": 28 + f, "autotune_timings": [[NOTE, f]] * 10}
                      for k in ("batched", "scaled_up_plain", "scaled_up_int8")},
        "delivery_saturating": {"kernel": "k_deliver_slices", "note": NOTE, "points": plain,
                                **{k: {"kernel": "k", "note": NOTE, "points": plain}
                                   for k in ("blocked6", "blocked4", "blocked8")},
                                "block_major": {"note": NOTE, "points": points}},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 6, "power_w_mean": 175.2266666666},
        "build_s": 1.655473024,
        "energy": {"joules": 20.329, "power_w_mean": 338.33, "nj_per_event": 9.899652242489616, "source": NOTE},
        "cpu_baseline": {"value": 43404683.21144581, "unit": "synaptic events/s", "cores": 1, "kind": "oracle",
                         "sample": NOTE, "rtf": 22.96, "multithreaded": {"value": 5.1e8, "cores": 16, "rtf": 1.93}},
    }


def test_line_is_short_and_whole():
    rec = _record()
    text = json.dumps(bench.headline(rec))
    line = json.loads(text)
    assert len(text) < 2800
    for key in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype",
                "data", "config", "gpu_launches"):
        assert line[key] == rec[key]
    assert line["value"] == pytest.approx(rec["value"], rel=1e-7)
    assert line["ms_per_step"] == pytest.approx(rec["ms_per_step"], rel=1e-7)
    assert set(line["e2e"]) == {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert line["clocks"]["reasons"] == [] and line["clocks"]["sm_mhz"] == 2070.0
    assert line["roofline"]["kernel"] == "k_step" and line["roofline"]["traffic"] == 1161472
    assert set(line["longest_lists"]) == {"rows", "blocked6", "blocked4", "blocked8", "block_major"}


def test_sections_that_a_run_leaves_out():
    rec = _record()
    rec.update(instances=None, compressed_records={}, workloads={},
               delivery_saturating={"points": [], "block_major": {"points": []}, "blocked6": {"points": None}})
    del rec["cpu_baseline"], rec["energy"]
    line = bench.headline(rec)
    assert line["longest_lists"] == {} and "cpu_baseline" not in line and line["ms_per_step"] > 0
