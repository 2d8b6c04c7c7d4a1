"""The benchmark's printed line (CPU): short enough for a log that keeps only the
end of the output, whatever was measured beside the result."""
import json

import bench


def _full(n_extra):
    prec = {k: {"ms": 18.123456789, "pts_per_s": 3482890.123456, "variant": "integer limbs", "imad_frac": 0.3380721,
                "out_GB_per_s": 61.2, "fp64_bodies": {"ms": 23.3, "pts_per_s": 2.8e6, "fp64_frac": 0.73}}
            for k in ("D", "DD", "QD")}
    work = {"paths": 65536, "plain_paths_per_s": 32923.61234, "learned_paths_per_s": 39850.312345,
            "speedup": 1.210391234, "train": {"note": "x" * 300}, "counts": {"plain": {"converged": 65536}}}
    return {"metric": bench.METRIC, "value": 613534.315944473, "unit": "pts/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 106.81717109680176, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64 (D, DD, QD limbs)", "data": "synthetic",
            "config": {"workload": "evaldiff_n32", "n_vars": 32, "note": "y" * 250}, "per_precision": prec,
            "tuned": {k: {"variant": "integer limbs", "threads": 256} for k in prec},
            "unfused_ablation": {"rows": ["z" * 100] * 14}, "paper_shapes": [{"a": 1.0 / 3}] * 400,
            "tracking": {"workload_%d" % k: work for k in range(n_extra)},
            "roofline": {"bound": "alu", "achieved": 4.96652, "peak": 8.4798, "frac": 0.58, "what": "w" * 200},
            "peaks": {"fp64_instr_per_s": 6.2e11}, "cpu_baseline": {"value": 94.3659, "sample": "s" * 80,
                                                                    "single_thread": {"value": 6.1}},
            "e2e": {"value": 263277.0884228, "unit": "pts/s", "h2d_bytes_per_step": 234881024,
                    "d2h_bytes_per_step": 7751073792, "ms_per_precision": {k: [1.5, 3.25, 2.0] for k in prec}},
            "gpu_launches": 60, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 20},
            "wall_s_timed_region": 2.1}


def test_line_is_short_and_complete():
    for n_extra in (0, 6, 40):  # 40: more than fit, dropped before anything that the result needs
        full = _full(n_extra)
        line = bench.result_line(full)
        assert len(line) <= bench.LINE_MAX and "\n" not in line
        d = json.loads(line)
        for k in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype",
                  "data", "config", "gpu_launches", "clocks"):
            assert d[k] == full[k], k
        for k in ("value", "ms_per_step"):
            assert abs(d[k] - full[k]) <= 1e-5 * full[k]
        e = d["e2e"]
        assert e["h2d_bytes_per_step"] == 234881024 and e["d2h_bytes_per_step"] == 7751073792
        assert e["ms_min_max"]["DD"] == [1.5, 3.25]
        assert (len(d.get("tracking", {})) == n_extra) == (n_extra <= 6)


def test_line_without_the_optional_measurements():
    full = _full(0)
    full.update(e2e=None, cpu_baseline=None, tracking={}, paper_shapes=None, unfused_ablation=None)
    d = json.loads(bench.result_line(full))
    assert d["e2e"] is None and d["value"] > 0
