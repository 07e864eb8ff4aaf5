"""The line that bench.py prints is read from the last kilobytes of a log: it stays short however much the run measures, and
keeps what its readers rely on."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def test_the_printed_line_is_short():
    import bench
    import paper_2503_23956_b200 as ac
    wl = bench.pick_workload("c5", None)
    number = 123456.78901234567
    stages = dict(score=number, budget=number, compact=number, decode=number)
    m = dict(stage_ms=stages, valid_rows=10 ** 9)
    roof, comp, score = bench.rooflines(ac, wl, m, 2, 256, traffic=number * 1e6)
    result = dict(metric=bench.METRIC, value=number, unit=bench.UNIT, n_gpus=8, steps=20, warmup=5, ms_per_step=number,
                  higher_is_better=True, scaling="weak", vs_baseline=None, dtype="bf16", data="synthetic",
                  config=bench.config_of(ac, wl, 1024, 2), decode_tok_s=number, compress_us_per_layer=number,
                  stage_us_per_request=stages, roofline=roof, roofline_compact=comp, roofline_score=score,
                  clocks=dict(sm_mhz=1965.0, sm_max_mhz=1965.0, reasons=["sw_power_cap"], samples=4000, detail=["x" * 500]),
                  gpu_launches=10 ** 6, e2e=dict(value=number, unit=bench.UNIT, ms_per_step=number, requests_per_step=1,
                                                 h2d_bytes_per_step=10 ** 11, d2h_bytes_per_step=10 ** 11,
                                                 api="aircache_pipeline_host", v_read_in_place=True),
                  workloads={str(i): dict(roofline=roof) for i in range(20)},
                  cpu_baseline=dict(value=number, unit=bench.UNIT, cores=16, kind="oracle", sample="y" * 300))
    line = json.dumps(bench.short_line(result), separators=(",", ":"))
    assert len(line) <= 1500, len(line)
    back = json.loads(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "roofline", "clocks", "gpu_launches", "e2e", "cpu_baseline"):
        assert key in back, key
    assert set(back["clocks"]) == {"sm_mhz", "sm_max_mhz", "reasons"}
    assert back["roofline"]["traffic"] == number * 1e6 and back["e2e"]["h2d_bytes_per_step"] == 10 ** 11
    assert "workloads" not in back and "roofline_score" not in back
