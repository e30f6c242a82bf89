"""The line bench.py prints stays short enough to be read whole: the headline's
keys as measured, one figure per further leg."""
import json

import bench


def _line(legs):
    roof = {"bound": "hbm", "achieved": 5712.123456789, "peak": 6677.2, "unit": "GB/s", "frac": 0.8554, "alg_bytes": 1}
    loop = {f"{k}@{r}": {"requests": 20000, "p50_ms": 0.0746612345, "p99_ms": 0.399916, "qps": 200.1033096, "failed": 0,
                         "batched_launches": 15, "requests_per_launch": 133.333}
            for k in ("served", "plain") for r in (200, 500, 1000, 2000, 5000)}
    loop["served@max"] = {"requests": 20000, "qps": 47649.49610085999}
    e2e = {"value": 1.9e10, "unit": "fact rows/s", "h2d_bytes_per_step": 570_000_000, "d2h_bytes_per_step": 16800,
           "raw_pages": {"value": 1e9}, "source": "pinned page pool, 64 MiB pages"}
    return {"metric": bench.METRIC, "value": 145273380946.1135, "unit": "fact rows/s", "n_gpus": 1, "steps": 20,
            "warmup": 5, "ms_per_step": 0.413, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "int64", "data": "synthetic", "config": {"workload": bench.WORKLOAD, "fact_rows": 60_000_000},
            "hbm_gbs": 5700.0, "roofline": roof, "e2e": e2e, "gpu_launches": 60,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "cpu_baseline": {"value": 1.6e7, "cores": 16, "sample": "x" * 150, "single_core": {"value": 1e6}},
            "extra": {f"leg-{i}": {"on": {"ms_per_step": 1.0 + i, "roofline": roof, "text": "y" * 300}}
                      for i in range(legs)},
            "patterns": {"batched": {"batched_ms": 1.07, "plain_ms": 18.5, "roofline": roof, "how": "z" * 300},
                         "served": {"requests_per_rate": "min(20000, 10 s x rate)", **loop}, "served_streamed": loop}}


def test_line_is_short_and_keeps_the_headline():
    line = _line(12)
    assert len(json.dumps(line)) > bench.LINE_BYTES
    out = json.loads(json.dumps(bench.brief(line)))
    assert len(json.dumps(out)) <= bench.LINE_BYTES
    for k in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "dtype", "config",
              "gpu_launches", "clocks"):
        assert out[k] == line[k]
    assert out["value"] == line["value"] and out["ms_per_step"] == line["ms_per_step"]
    assert out["e2e"]["h2d_bytes_per_step"] == line["e2e"]["h2d_bytes_per_step"]
    assert out["extra"]["leg-3"] == {"ms": 4.0}
    assert out["patterns"]["served"]["plain@500"] == [0.0746612, 0.399916]
    assert out["patterns"]["served"]["served@max"] == 47649.5


def test_headline_survives_any_number_of_legs():
    out = bench.brief(_line(400))
    assert len(json.dumps(out)) <= bench.LINE_BYTES
    assert out["e2e"]["unit"] == "fact rows/s" and out["roofline"]["frac"] == 0.8554
