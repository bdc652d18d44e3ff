"""The benchmark's printed line: the keys its readers need, short enough that the end
of a captured output holds all of it, whatever the phases' records hold."""
import json


def _record():
    long = {"note": "x" * 5000, "rows": list(range(2000))}
    rec = {k: 1.0 for k in ("value", "n_gpus", "steps", "warmup", "ms_per_step", "gpu_launches", "wall_s_timed")}
    rec.update(metric="m", unit="u", higher_is_better=True, scaling="weak", vs_baseline=None, dtype="f32",
               data="synthetic", config={"workload": "w" * 150, "S": 256}, clocks={"sm_mhz": 2070.0, "reasons": []},
               untuned={"value": 1.0, "config": "c"}, roofline={"bound": "alu", "achieved": 1.0, "frac": 0.1, **long},
               e2e={"value": 2.0, "unit": "u", "h2d_bytes_per_step": 3, "d2h_bytes_per_step": 4, **long},
               cpu_baseline={"value": 1.0, "unit": "u", "cores": 16, "kind": "oracle", **long})
    rec.update({k: long for k in ("tuning", "stream", "c2", "batched", "gemm_dynamic", "precision")})
    return rec


def test_line_is_short_and_whole():
    import bench
    rec = _record()
    text = json.dumps(bench.headline(rec))
    assert len(text) < 1500
    line = json.loads(text)
    for key in bench.HEADLINE:
        assert line[key] == rec[key]
    assert line["e2e"] == {"value": 2.0, "unit": "u", "h2d_bytes_per_step": 3, "d2h_bytes_per_step": 4}
    rec["cpu_baseline"] = None
    assert bench.headline(rec)["cpu_baseline"] is None
