"""The result line of bench.py stays short enough to be read whole from a log's tail: the
tables by point and the legs' details are printed apart."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

X = 123456789.12345679
ROOF = {"bound": "alu", "achieved": X, "peak": X, "unit": "Tlane-op/s", "frac": 0.123456789012, "traffic": X,
        "traffic_unit": "bytes per launch", "algorithmic_bytes_per_launch": 123456789, "nms_ms_per_step": X,
        "kernel": "bch_nms_jit + bch_nms_rc", "lane_ops_per_edge_update": 8, "edge_updates_per_s": X,
        "peak_basis": "152 SMs x 128 lanes x 2070 MHz (median SM clock under load)", "ld": 64}
POINT = {"code": "(63,36)", "ebn0": 1.0, "frames": 10 ** 6, "fer": X, "fer_ci95": [X, X], "ber": X, "osd_frames": 10 ** 6,
         "nms_fer": X, "avg_iters": X, "iters_hist": [10 ** 6] * 12, "undetected": 10 ** 6, "oracle_fer": X,
         "oracle_ci95": [X, X], "gpu_fer_on_oracle_frames": X}
SERVED = {k: X for k in ("requests", "frames", "frame_errors", "p50_ms", "p99_ms", "mean_ms", "max_ms", "elapsed_s",
                         "served_frames_per_s", "offered_frames_per_s", "offered_requests_per_s")}
RATE = {"rate_rps": X, "server": SERVED, "static_batching": SERVED}
PHASE = {k: X for k in ("ms_wall", "ms_h2d", "ms_decode", "ms_d2h")}


def _line():
    return {"metric": bench.METRIC, "value": X, "unit": "frames/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": X, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": {"workload": "w" * 150, "codes": ["(63,36)", "(63,45)"]},
            "edge_updates_per_s": X, "roofline": ROOF, "cpu_baseline": {"value": X, "sample": "s" * 120},
            "e2e": {"value": X, "unit": "frames/s", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1, "mode": "m" * 120,
                    "phases_per_code_call": [PHASE] * 2, "staged_copies": {"value": X, "phases_per_code_call": [PHASE] * 2}},
            "clocks": {"sm_mhz": X, "sm_max_mhz": X, "reasons": [], "samples": 9}, "gpu_launches": 999,
            "msg_legs": {k: {"frames_per_s": X, "ms_per_step": X, "roofline": ROOF, "frame_errors_per_code": [1, 2]}
                         for k in ("fp16", "int8", "int8f")},
            "config4": {"workload": "w" * 120, "frames_per_step": 10 ** 7, "frames_per_s": X, "ms_per_step": X,
                        "codes": {k: {"roofline": ROOF, "per_point": [POINT] * 7} for k in ("(127,64)", "(127,99)")}},
            "pcm_search": {"workload": "w" * 90, "chains": 1216, "search_s": X, "four_cycles": {"chain0": 1, "kept": 1},
                           "nms_fer_at_3dB": {"chain0": POINT, "kept": POINT}},
            "serving": {"workload": "w" * 120, "seconds": 10.0, "server_kernel": "jit", "server": SERVED,
                        "static_batching": SERVED, "below_saturation": RATE, "twice_the_rate": RATE,
                        "static_batching_plain_nms": {"config_rate": SERVED, "below_saturation": SERVED},
                        "server_stats": SERVED},
            "training": {"workload": "w" * 90, "steps": 20, "ms_per_step": X, "frames_per_s": X, "loss_first": X,
                         "loss_last": X, "alpha": [X] * 12},
            "plain_nms": {"workload": "w" * 120, "frames_per_s": X, "us_per_decode": X, "fer": X, "ber": X},
            "fer_match_oracle_ci95": True, "fer_match_detail": {"points": 22}, "per_point": [POINT] * 22}


def test_line_is_short_and_loses_nothing():
    full = _line()
    short, tables = bench.headline(full)
    assert len(json.dumps(full)) > 15_000 and len(json.dumps(short)) < 6_000
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "roofline", "cpu_baseline", "e2e", "clocks", "gpu_launches",
                "fer_match_oracle_ci95"):
        assert short[key] == full[key]
    assert all(tables[k] == full[k] for k in full if k not in short or short[k] != full[k])
    assert short["serving"]["server"]["p99_ms"] == X and short["config4"]["codes"]["(127,64)"]["frac"] == ROOF["frac"]


def test_legs_that_were_skipped_or_failed():
    short, _ = bench.headline({**_line(), "config4": None, "pcm_search": None, "serving": {"error": "closed"},
                               "training": None, "plain_nms": None, "msg_legs": {}})
    assert short["serving"] == {"error": "closed"} and short["training"] is None and short["msg_legs"] == {}


def test_traffic_belongs_to_the_kernel_that_ran(monkeypatch):
    """A launch's DRAM traffic is scaled from a capture of the same kernel, block length and
    format, and left out where there is none."""
    import types
    props = types.SimpleNamespace(multi_processor_count=152)
    torch = types.SimpleNamespace(cuda=types.SimpleNamespace(get_device_properties=lambda dev: props))

    def traffic(kernel, n, fp32=True):
        return bench.nms_roofline(torch, 0, {"sm_mhz": 2070.0}, 1e9, 1e-3, kernel, 1000, n, fp32=fp32)["traffic"]

    assert traffic("bch_nms_jit + bch_nms_rc", 63) == 1000 * bench.DRAM_BYTES_PER_FRAME["bch_nms_jit", 63]
    assert traffic("bch_nms_rc", 127) == 1000 * bench.DRAM_BYTES_PER_FRAME["bch_nms_rc", 127]
    assert traffic("bch_nms_rc", 63) is None and traffic("bch_nms_jit", 127) is None
    assert traffic("bch_nms_jit", 63, fp32=False) is None and traffic("nms_enhanced_kernel", 63) is None
