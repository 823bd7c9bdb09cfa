"""The bench's printed line: the headline keys and one figure per configuration, short enough to be
read back from the end of a log (host logic on a synthetic record, no GPU)."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def record():
    import bench
    kinds = [f"kind_{i}" for i in range(10)]
    serving = {arm: {"achieved_req_s": 1000.0, "p50_us": 8.0, "p99_us": 11.0, "parity_sample": "ok"}
               for arm in ("persistent", "persistent_device_ring", "per_request_launch")}
    return {
        "metric": bench.METRIC, "value": 880314.27, "unit": "acq/s", "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 403.7, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
        "data": "synthetic", "config": bench.step_config(1), "gpu_launches": 920,
        "e2e": {"value": 874504.1, "unit": "acq/s", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
        "roofline": {"frac": 0.7, "traffic_note": bench.ROOF_TRAFFIC_NOTE, "peak_source": "x" * 500},
        "cpu_baseline": {"value": 1.4e6, "sample": "x" * 200}, "parity_after_timing": "ok",
        "mutex": {k: {str(cs): {"acq_per_s": 812345.678, "roof_acq_per_s": 1e6, "frac": 0.8, "note": "x" * 300}
                      for cs in bench.CS_SIZES} for k in kinds},
        "barrier": {"kinds": {k: {"ns_per_crossing": 2068.123456, "roof_ns": 1200.0, "frac": 0.5, "note": "x" * 300}
                              for k in kinds + [k + "b" for k in kinds]}},
        "semaphore": {"kinds": {k: {n: {"ops_per_s": 3e5, "roof_ops_per_s": 4e5, "frac": 0.7} for n in ("1", "4", "16")}
                                for k in kinds[:4]}},
        "condvar": {"mutex": {k: {"items_per_s": 3e5, "frac": 0.48} for k in kinds[:4]}},
        "batched": {"default": {"acq_per_s": 4.8e6, "cluster": 1}, "tuned": {"acq_per_s": 5.2e6, "cluster": 4}},
        "serving": {"rates": {str(10 ** k): serving for k in (3, 4, 5, 6)}},
        "sweep": {"mutex_acq_per_s": {k: {"64": {str(B): 9e5 for B in range(1, 30)}} for k in kinds}},
        "roofline_terms": {f"term_{i}": 1.0 for i in range(300)},
    }


def test_line_is_short_and_holds_the_contract():
    import bench
    out = record()
    line = json.dumps(bench.headline(out))
    assert len(line) < 12_000 < len(json.dumps(out))
    got = json.loads(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert got[key] == out[key], key


def test_line_holds_one_figure_per_configuration():
    import bench
    out = record()
    got = bench.headline(out)["figures"]
    rows = [r for r in bench.result_rows(out) if not r["section"].startswith("sweep")]
    assert sum(len(v) for v in got.values()) == len(rows)
    assert got["acq_per_s"]["mutex kind_3 cs_words=64"] == 812350.0
    assert got["p99_us"]["serving persistent offered_req_s=100000"] == 11.0


def test_line_without_sections():
    import bench
    assert bench.headline({"value": 1.0, "config": {}, "n_gpus": 1}) == {"value": 1.0, "config": {}, "n_gpus": 1,
                                                                        "figures": {}}
