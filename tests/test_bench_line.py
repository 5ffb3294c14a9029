"""The line that bench.py prints: one JSON line on stdout that stays short however much was measured (a reader that
keeps the last few KB of a run has to find it whole), everything on stderr and in the file of --details."""
import json

import bench


def _line():
    variant = {"ms_per_step": 0.4812345678, "value": 2078.0, "roofline": {"note": "x" * 400}, "solver": "CG"}
    return {"metric": bench.METRIC, "value": 2095.0, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.4773, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": bench._labels("fp16", 1, 1)[0], "data": "synthetic (seeded)",
            "config": {"workload": bench.WORKLOAD, "precision": bench._labels("fp16", 1, 1)[1]},
            "roofline": {"bound": "hbm", "achieved": 808.4, "peak": 6748.3, "frac": 0.12},
            "e2e": {"value": 1167.0, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2, "note": "y" * 500},
            "gpu_launches": 60, "clocks": {"sm_mhz": 2070.0, "reasons": []},
            "c1_variants": {f"v{k}": dict(variant) for k in range(8)}, "c2_mixed": {"n": 1, **{f"w{k}": dict(variant) for k in range(6)}},
            "reduced_variant": dict(variant), "c3_batch": {"ms_per_launch": 51.3, "plan": "z" * 800}, "c0_l96": {"cycles_per_s": 1075.4},
            "e2b_table5": {"1000": {"enkf_reduced_ms": 0.25, "more": "q" * 900}, "note": "n"},
            "cpu_baseline": {"value": 3.4, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 200}}


def test_the_line_is_short_and_whole_and_the_rest_is_kept(capsys, tmp_path):
    line = _line()
    bench._emit(line, str(tmp_path / "d.json"))
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) <= 4096
    head = json.loads(out)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
              "dtype", "data", "config", "roofline", "gpu_launches", "clocks", "cpu_baseline"):
        assert k in head, k
    assert head["value"] == line["value"] and head["e2e"]["h2d_bytes_per_step"] == 1 and "note" not in head["e2e"]
    assert head["sections"]["c1_v0_ms"] == 0.4812 and head["sections"]["e2b_1000_ms"] == 0.25
    assert json.loads(err) == line and json.loads((tmp_path / "d.json").read_text()) == line


def test_a_line_without_sections_is_printed_once(capsys):
    line = {k: v for k, v in _line().items() if k in bench._LINE_KEYS}
    bench._emit(line)
    out, err = capsys.readouterr()
    assert err == "" and "sections" not in json.loads(out)


def test_labels_of_the_preconditioned_modes_name_the_solve_they_share():
    for prec in ("fp32", "fp16", "bf16"):
        for order in (0, 1):
            dtype, name, sums = bench._labels(prec, 1, order)
            assert dtype == "f32" and "exact FP16 slices" in name and sums == bench.REDUCE_NAME[0]
        assert bench._labels(prec, 0, 1)[0] == bench.DTYPE[prec] and bench._labels(prec, 0, 1)[2] == bench.REDUCE_NAME[1]
