"""The benchmark's result line: short enough for what keeps only the end of a run's
output, with everything the contract names (the whole record goes to --details)."""
import json

import bench


def _record():
    roofline = {"bound": "alu", "achieved": 7.761214323533427, "peak": 40.27392, "unit": "Tops/s", "frac": 0.1927106753,
                "traffic": None, "peak_source": "x" * 60, "msg_updates_counted": "x" * 140, "kernel": "k_round",
                "launch_ms": 5.448099211355051, "kernel_share": 0.7680810444604177, "measured_in": "x" * 110}
    form = {"value": 107631607.35496064, "unit": "syndromes/s", "ms_per_step": 2.787, "roofline": roofline,
            "per_p": {p: {"ler": 0.0, "seed_converged": 0.99, "mean_alg_iters": 1.06} for p in ("0.001", "0.002", "0.003")},
            "cpu_baseline": {"value": 8300.0, "unit": "syndromes/s"}}
    shapes = {p: {"group_warps": 1, "warps_per_block": 8, "sample_shots": 65536, "timed": [[1, 8, 0.2294]] * 8}
              for p in ("0.01", "0.03", "0.05")}
    return {
        "metric": bench.METRIC, "value": 140691742.8103948, "unit": "syndromes/s", "n_gpus": 1, "steps": 10, "warmup": 3,
        "ms_per_step": 21.323213005065917, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic", "config": {"workload": "w" * 70, "code": "c" * 40, "shots_per_p_per_gpu": 1000000,
                                        "l2": "l" * 70, "parallelism": "single GPU", "launch_shapes": shapes},
        "hbm": {"dram_gbs": None, "source": "s" * 100}, "roofline": roofline, "gpu_launches": 240,
        "per_p": {p: {"ler": 5e-06, "kernel_ms_per_step": {f"k{n}": 0.781190383434 for n in range(6)}} for p in shapes},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 3, "power_w_max": 261.22},
        "e2e": {"value": 135936587.8654959, "unit": "syndromes/s", "h2d_bytes_per_step": 36000000,
                "d2h_bytes_per_step": 96000000, "api": "bsd_decode_host (pinned host buffers)"},
        "cpu_baseline": {"value": 149714.16687, "unit": "syndromes/s", "cores": 16, "kind": "oracle", "sample": "s" * 100,
                         "single_core": {"value": 10249.3, "sample": "s" * 80}},
        "side_by_side": {"phenomenological_dem": {"forms": {f: dict(form) for f in ("fp32", "fp16", "bf16")}},
                         "synthetic_dem": {"value": 107471617.83, "per_width": {w: dict(form) for w in ("8", "32", "64")}}},
    }


def test_a_long_record_becomes_a_short_line(capsys, tmp_path, monkeypatch):
    line = _record()
    monkeypatch.setattr(bench, "DETAILS_FILE", str(tmp_path / "details.json"))
    bench.emit(line)
    got = capsys.readouterr()
    whole = (tmp_path / "details.json").read_text()
    assert json.loads(whole) == line and len(whole) > 6000
    assert got.err == "" and got.out.count("\n") == 1 and len(got.out) <= bench.LINE_LIMIT + 1
    out = json.loads(got.out)
    for key in bench.CONTRACT:
        assert (key in out) == (key in line or key == "ler"), key
    assert out["ler"] == {"0.01": 5e-06, "0.03": 5e-06, "0.05": 5e-06}
    for key in ("metric", "unit", "n_gpus", "steps", "warmup", "gpu_launches", "data", "dtype", "vs_baseline"):
        assert out[key] == line[key]
    assert abs(out["value"] / line["value"] - 1) < 1e-6 and abs(out["e2e"]["value"] / line["e2e"]["value"] - 1) < 1e-6
    assert out["clocks"]["sm_mhz"] == 2070.0 and out["clocks"]["reasons"] == []
    assert out["side_by_side"]["synthetic_dem"] == 1.0747e8
    assert out["side_by_side"]["phenomenological_dem.fp16"] == 1.0763e8


def test_a_short_line_is_left_alone(capsys):
    bench.emit({"impl": "reference", "value": 1.0 / 3.0})
    got = capsys.readouterr()
    assert json.loads(got.out) == {"impl": "reference", "value": 1.0 / 3.0} and got.err == ""
