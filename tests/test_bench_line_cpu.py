"""The line that bench.py prints stays short enough to be kept whole by a reader
of the last few thousand characters of its output, with every leg run, and
carries the headline as measured; the full record goes to a file."""
import importlib
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


CONFIG = ("va_edge_pre=128t,va_cell_vert=512,column_threads=160;column_columns=32;column_corrector_threads=160;"
          "column_corrector_chunk=4;column_chunk=8")


def _full(B):
    """A record of a default run: kernel tables of the real kernels, long numbers, notes."""
    x = 1234.567890123456789
    nc, ne, nv = 327680, 491520, 163842
    prof = {k: (10, x / 100) for k in B.FLOPS_PER_UNIT}
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 123}
    hbm = {"bytes_per_step": x * 1e9, "achieved_gbs": x, "peak_gbs": x, "peak_source": "measured", "frac": x / 3000,
           "stage_bytes_per_step": x * 1e9, "amplification": x / 1000, "note": "n" * 200}
    leg = {"value": x, "ms_per_step": x, "speedup_vs_fp64": x / 999, "finite": True, "rms_ps_pa": x * 1e-7,
           "rms_t850_k": x * 1e-9, "reference": "r" * 200, "hbm_measured": hbm, "kernels": B.kernel_table(prof, 2),
           "clocks": clocks, "autotuned_launch_config": "a" * 600, "sdpd": x}
    learned = dict(leg, fallbacks_timed=0, rms_ps_pa_vs_fp64=x, train={"seconds": x}, error_vs_plain_step={"a": x})
    return {
        "metric": B.METRIC, "value": x / 100, "unit": "steps/s", "n_gpus": 8, "steps": 100, "warmup": 100,
        "ms_per_step": x, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": B.config_dict("fp64"), "sdpd": x, "hbm": dict(hbm, stage_frac=x),
        "hbm_measured": hbm, "roofline": B.roofline(prof, nc, ne, nv, 90, chunks=B.column_chunks(CONFIG)), "kernels": B.kernel_table(prof, 2),
        "autotuned_launch_config": "a" * 600, "steps_compared": 240, "mixed": leg, "mixed_f64col": leg,
        "mixed_learned": learned, "mountain_r2b7": {"config": {}, "fp64": leg, "mixed": leg, "mixed_learned": learned},
        "e2e": B.end_to_end([x / 1000] * 9 + [x / 500], 1536163840),
        "gpu_launches": 123456, "clocks": clocks, "finite": True,
        "cpu_baseline": {"value": x, "unit": "steps/s", "cores": 16, "kind": "oracle", "sample": "s" * 400,
                         "extrapolated": True, "single_thread": {"value": x}}}


def test_the_line_of_a_default_run_is_short_and_whole():
    if ROOT not in sys.path:
        sys.path.insert(0, ROOT)
    B = importlib.import_module("bench")
    full = _full(B)
    text = json.dumps(B.result_line(full))
    assert len(text) <= B.LINE_LIMIT, len(text)
    line = json.loads(text)
    for k in B.LINE_KEYS:
        assert line[k] == full[k], k
    for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][k] == full["e2e"][k], k
    for k in ("mixed", "mixed_f64col", "mixed_learned"):
        assert abs(line[k]["value"] / full[k]["value"] - 1.0) < 1e-4
        assert abs(line[k]["hbm_frac"] / full[k]["hbm_measured"]["frac"] - 1.0) < 1e-4
        assert abs(line["mountain_r2b7"][k if k != "mixed_f64col" else "fp64"]["value"] / full[k]["value"] - 1.0) < 1e-4
    assert abs(line["hbm_measured"]["frac"] / full["hbm_measured"]["frac"] - 1.0) < 1e-4


def test_the_line_of_a_run_without_legs():
    if ROOT not in sys.path:
        sys.path.insert(0, ROOT)
    B = importlib.import_module("bench")
    full = _full(B)
    for k in ("hbm", "hbm_measured", "roofline", "kernels", "mixed", "mixed_f64col", "mixed_learned", "mountain_r2b7",
              "e2e", "clocks", "finite", "value", "ms_per_step"):
        full[k] = None
    full.pop("cpu_baseline")
    line = json.loads(json.dumps(B.result_line(full)))
    assert line["value"] is None and line["e2e"] is None and "mixed" not in line


def test_the_end_to_end_rate_counts_every_step():
    if ROOT not in sys.path:
        sys.path.insert(0, ROOT)
    B = importlib.import_module("bench")
    e = B.end_to_end([0.1] * 8 + [0.165, 0.164], 7)
    assert abs(e["value"] - 10 / (0.8 + 0.165 + 0.164)) < 1e-12
    assert abs(e["median_value"] - 10.0) < 1e-12
    assert e["h2d_bytes_per_step"] == e["d2h_bytes_per_step"] == 7 and e["step_ms"][-2:] == [165.0, 164.0]


def test_fp64_instructions_are_those_of_the_chunks_that_ran():
    if ROOT not in sys.path:
        sys.path.insert(0, ROOT)
    B = importlib.import_module("bench")
    nc, ne, nv = 327680, 491520, 163842
    prof = {"sn_column_pred": (5, 10.0), "sn_column_corr": (5, 12.0)}
    t = B.FP64_INSTR_PER_UNIT
    for corr in (4, 6, 8):
        text = CONFIG.replace("corrector_chunk=4", "corrector_chunk=%d" % corr)
        r = B.roofline(prof, nc, ne, nv, 90, chunks=B.column_chunks(text))
        want = (t["sn_column_pred"][8] + t["sn_column_corr"][corr]) * nc * 90 * 5 / 0.022 / 1e12
        assert abs(r["fp64_issue"]["achieved"] - want) < 1e-12 * want
    assert B.column_chunks(CONFIG.replace("columns=32", "columns=16")) == {}
    assert B.roofline(prof, nc, ne, nv, 90, chunks={})["fp64_issue"] is None
