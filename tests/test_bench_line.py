"""What the benchmark prints and searches (CPU only)."""
import json

import pytest

pytest.importorskip("torch")


def _result():
    """A whole result with every part as large as a run makes it."""
    import bench
    from paper_2408_02367_gb300 import synth
    w = synth.WORKLOADS["vol128_w4"]
    f = 0.12345678901234567
    tuning = {"spread_bins": [4, 4, 4], "spread_chunk": 512, "fft_engine": 0, "fft_lines": 0, "fft_cols": 0, "interp_threads": 256,
              "spread_coils": 0, "interp_run": 1, "interp_coils": 0, "fft_staged": 3, "interp_tiled": 1}
    table = [{"tuning": tuning, "ms": f, "rel_vs_first": f}] * 20
    orc = bench.oracle_line(w, 2, [f, f], 10, "bench workload")
    stages = {k: f for k in bench.stage_bytes(w, 2, (160, 160, 160), 1000)}
    roof = {"bound": "hbm", "kernel": "adj_ifft3_epilogue", "achieved": f, "peak": f, "unit": "GB/s", "frac": f, "peak_kind": "measured",
            "traffic": f, "alg_bytes_per_launch": f, "avg_launch_ms": f, "launches_per_step": f}
    return {"metric": bench.METRIC, "value": f, "unit": bench.UNIT, "n_gpus": 1, "steps": 400, "warmup": 10, "ms_per_step": f,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": bench.workload_desc(w, 2), "grid": [160] * 3, "l2": "x" * 70, "timed": "x" * 80,
                       "parallelism": "single GPU", "coil_draws": "x" * 70},
            "dip_step_ms": {"eager": f, "cuda_graph": f}, "plain_form": {k: f for k in "abcde"}, "roofline": roof,
            "stage_ms_per_step": stages, "stage_share": stages, "stage_roofline": {k: roof for k in stages},
            "path_model": {"bytes_per_step": f, "frac_of_hbm_bound": f}, "operator_rows": {str(i): f for i in range(40)},
            "scale_rows": {"whole_brain": {"autotuner": table}, "multi_volume": {"volumes": table}},
            "tuning": {"chosen": tuning, "autotuner": table, "note": "x" * 130},
            "cpu_baseline": dict(orc, other_workloads={"vol32_w6": orc}),
            "e2e": {"value": f, "unit": bench.UNIT, "h2d_bytes_per_step": 91750408, "d2h_bytes_per_step": 83886084, "ms_per_step": f,
                    "steps": 50, "serial_ms_per_step": f, "note": "x" * 300},
            "gpu_launches": 3600, "gpu_launches_eager_region": 3600, "clocks": {"sm_mhz": f, "sm_max_mhz": f, "power_w_max": f,
                                                                               "reasons": ["sw_power_cap"], "samples": 20}}


def test_printed_line_is_short_and_whole():
    """A reader takes the line from the last few kilobytes of stdout: with the tables in it, 27 KB, it was
    never read.  It keeps every key of the benchmark's contract, and the details keep the rest."""
    import bench
    full = _result()
    line, details = bench.split_result(full)
    assert len(json.dumps(line)) < 4096 < len(json.dumps(details))
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
              "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert k in line
    assert line["e2e"] == full["e2e"] and line["tuning"]["chosen"] == full["tuning"]["chosen"]
    assert set(full) == set(line) | (set(details) - {"tuning_autotuner", "cpu_baseline_other_workloads"})
    assert details["tuning_autotuner"] == full["tuning"]["autotuner"]
    assert "autotuner" in full["tuning"]           # the result itself is left as it was


def test_measured_traffic_of_tunings_that_differ_without_effect():
    import bench
    t = {"spread_bins": (8, 4, 4), "interp_tiled": 1, "fft_staged": 3, "fft_cols": 0}
    assert bench.kernel_variant(t) == {"spread_bins": [4, 4, 4], "interp_tiled": 1, "fft_staged": 3, "fft_cols": 32}
    assert bench.kernel_variant(dict(t, spread_bins=(8, 4, 8)))["spread_bins"] == [4, 4, 8]


def test_no_two_candidates_are_the_same_kernels():
    """Every candidate of the autotuner (each builds a plan and is timed) differs from the others in a
    knob that chooses a kernel, in both rounds and for the bench's whole-brain lists."""
    import bench
    from paper_2408_02367_gb300 import tune

    def kernels(t):
        t = dict(tune.DEFAULT, **t)
        rows = () if t["interp_tiled"] else (t["interp_threads"] or 256, t["interp_run"] or 1, t["interp_coils"])
        return (t["spread_bins"][2], min(t["spread_chunk"], 512), t["spread_coils"] == 1, t["fft_engine"], t["fft_staged"],
                t["interp_tiled"], rows)

    for first, variants in ((tune.candidates(), tune.REFINE), (tune.candidates(full=True), tune.REFINE),
                            (bench.WHOLE_BRAIN_CANDIDATES, bench.WHOLE_BRAIN_REFINE)):
        assert len({kernels(t) for t in first}) == len(first)
        for base in first:
            second = tune.refinements(dict(tune.DEFAULT, **base), variants)
            assert len({kernels(t) for t in second}) == len(second)
