"""The bench's one line stays within what its readers keep of it."""
import json

import bench


def _record():
    curve = [[0.01 * i, 20.0 + 0.123456789 * i] for i in range(41)]
    runs = {k: {"psnr_curve": curve, "fallbacks": 0} for k in ("jacobi", "learned", "block_jacobi")}
    text = "a long explanation of what was counted and how, repeated until it is long enough " * 4
    return {"metric": "PCG iters/s", "value": 19.123456789012345, "unit": "PCG iters/s", "n_gpus": 1, "steps": 20,
            "warmup": 5, "ms_per_step": 2612.123456789, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic (seeded)",
            "config": {"workload": "scale128", "n_rays": 64000000, "tuning": {"tile_w": 8, "tile_h": 4}},
            "gpu_launches": 4355, "rays_per_s": 2.5e9,
            "gn_steps": [{"F_before": 1.0, "F_after": 0.5}] * 20,
            "roofline": {"bound": "alu", "achieved": 19.5, "peak": 80.5, "frac": 0.2423456789, "traffic_source": text,
                         "atomics": {"what": text, "frac": 0.89}, "design_traffic": {"what": text}},
            "vector_roofline": {"frac": 0.6, "note": text}, "residual_roofline": {"frac": 0.1, "note": text},
            "e2e": {"value": 18.5, "unit": "PCG iters/s", "h2d_bytes_per_step": 807845888, "d2h_bytes_per_step": 1},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "cpu_baseline": {"value": 0.02, "sample": text},
            "lpc": {"training": {"x": 1}, "gn": {"paper": {"runs": runs}, "fixed2": {"runs": runs}},
                    "summary": {"paper": {"learned": 0.5}, "fixed2": {"learned": 1.09}}}}


def test_long_record_is_cut_and_keeps_the_contract():
    line = _record()
    assert len(json.dumps(line)) > 2 * bench.LINE_LIMIT
    kept = bench.kept_line(line)
    assert len(json.dumps(kept)) <= bench.LINE_LIMIT < 3000
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "gpu_launches", "config", "e2e", "clocks"):
        assert kept[k] == line[k], k
    assert kept["roofline"]["bound"] == "alu"
    assert "psnr_curve" not in json.dumps(kept)


def test_short_record_is_printed_as_it_is(capsys):
    line = {k: v for k, v in _record().items() if k not in ("lpc", "roofline", "gn_steps", "vector_roofline",
                                                            "residual_roofline", "cpu_baseline")}
    assert bench.kept_line(line) is line
    bench.emit(line)
    out, err = capsys.readouterr()
    assert json.loads(out) == line and out.count("\n") == 1 and not err


def test_long_record_goes_whole_to_stderr(capsys):
    bench.emit(_record())
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) <= bench.LINE_LIMIT + 1
    assert json.loads(err.removeprefix("bench record: ")) == _record()
