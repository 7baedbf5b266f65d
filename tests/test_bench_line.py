"""The bench's record line: all keys of the contract, short enough to be read from the end of a log."""
import json

import bench


def test_the_record_line_is_short_and_has_its_keys():
    ops = {n: [6123.456789, 0.76543] for n in ("store_raw", "retrieve_raw", "compose_raw", "store_int8", "retrieve_int8", "compose_int8")}
    rec = {
        "metric": bench.METRIC, "value": 5987.654321987, "unit": bench.UNIT, "n_gpus": 8, "steps": 20, "warmup": 5, "ms_per_step": 12.3456789012,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16/int8 (fp32 codec and rotation, fp64 angles)", "data": "synthetic",
        "tokens_per_s_reloaded": 123456789.123, "gpu_launches": 1234, "config": {"workload": bench.WORKLOAD, "l2": "x" * 60, "bytes_per_step": 1 << 40, "also_measured": "y" * 500},
        "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "power_w_max": 900.0, "samples": 9, "reasons": ["sw_power_cap"]},
        "e2e": {"value": 51.23456789, "unit": "GB/s", "h2d_bytes_per_step": 1 << 36, "d2h_bytes_per_step": 1 << 36, "steps": 4, "ms_per_step": 345.6789,
                "host_link_gbs": 50.1, "host_link_peak": {"h2d_gbs": 55.0}, "what": "z" * 80},
        "cpu_baseline": {"value": 3.2, "unit": "GB/s", "cores": 16, "kind": "oracle", "sample": "s" * 130, "one_core": {}},
        "roofline": {"bound": "hbm", "kernel": "k" * 60, "op": "compose_int8", "achieved": 6123.456, "peak": 6452.2, "peak_kind": "of measured", "unit": "GB/s",
                     "frac": 0.94912345, "traffic": 1234567.0, "note": "n" * 300, "per_op": {"8b": ops, "70b": ops, "fractions": "f"}},
        "ops": {"filler": "o" * 20000},
    }
    line = bench.record_line(rec)
    assert "\n" not in line and len(line) <= bench.LINE_MOST
    got = json.loads(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config",
                "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline", "gbs_8b", "gbs_70b"):
        assert key in got, key
    assert got["value"] == 5987.65 and got["e2e"]["h2d_bytes_per_step"] == 1 << 36 and got["clocks"]["reasons"] == ["sw_power_cap"]
    rec["roofline"]["kernel"] = "k" * 2000                                     # what is optional goes before the line gets longer
    assert "gbs_8b" not in json.loads(bench.record_line(rec))
