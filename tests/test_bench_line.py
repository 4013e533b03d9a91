"""bench.py's result line stays short whatever the secondary workloads add, and
the pin that it reports rebuilds the launch configuration."""
import json

import bench

STRIPS = dict(strategy=1, block=800, tma=1, tile=4096, stages=6, lanes_per_row=8, map=1, col_map=0,
              transposed_rows=116612, scatter_patch=1)


def _record():
    kernels = {f"kernel {k}": {"ms_per_sweep": 1 / 3, "gbs_alg": 1e4 / 3} for k in range(4)}
    shape = dict(STRIPS, pin=bench.pin_of(STRIPS), tiles=0)
    solve = {"solves_per_s": 66.123456789, "p50_s": 1 / 3, "p99_s": 2 / 3, "formats": {"x": "f16"}}
    return {"metric": "m", "value": 1e12 / 3, "unit": "u", "n_gpus": 1, "steps": 10, "warmup": 3, "ms_per_step": 1 / 3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"model": "x" * 300}, "roofline": {"note": "y" * 400}, "kernels": kernels,
            "e2e": {"value": 1.0, "unit": "u", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2},
            "gpu_launches": 5, "clocks": {"sm_mhz": 2070, "sm_max_mhz": 2070, "reasons": []}, "launch_shape": shape,
            "variants": {f"a_workload_of_a_long_name_{k}": {"value": 1e12 / 7, "kernels": kernels} for k in range(20)},
            "precision": {f"p{k}": {"q" * 40: 1 / 3} for k in range(30)},
            "serving": {"requests": 512, "batched": solve, "single": solve, "mix": {"a": 1}},
            "cpu_baseline": {"value": 1.0, "unit": "u", "cores": 16, "kind": "oracle", "sample": "z" * 400}}


def test_the_line_is_short_and_complete():
    rec = _record()
    line = bench.headline(rec)
    assert len(json.dumps(line)) < 4096 < len(json.dumps(rec))
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline"):
        assert line[k] == rec[k], k
    assert line["launch_shape"]["pin"] == "1,0,0,0,0,0,0" and "tiles" not in line["launch_shape"]
    assert len(line["variants"]) == 20 and line["serving"]["batched"]["p50_s"] == 0.3333


def test_the_pin_of_a_form_asks_for_that_form():
    o = bench.pinned_opts(None, bench.pin_of(STRIPS))
    assert o == dict(strategy=1, stream_shape=(0, 0, 0), stream_map=0, stream_col_map=0, scatter_transpose=0)
    streamed = dict(STRIPS, block=768, lanes_per_row=32, map=2, transposed_rows=5)
    assert bench.pin_of(streamed) == "1,4096,6,32,2,0,2"
    assert bench.pin_of(dict(streamed, scatter_patch=0)) == "1,4096,6,32,2,0,1"
    assert bench.pin_of(dict(streamed, strategy=2, col_map=1, transposed_rows=0)) == "2,4096,6,32,2,1,-1"
