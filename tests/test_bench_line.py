"""The bench's result line stays short enough to be read whole from the end of a
log, its tables come on lines of their own, and the prediction's kernel is held
against the peak of the pipe it runs on.  No GPU."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def full_line():
    rows = [{"level": m, "stage": "aggregate", "kernel": "k" * 24, "ms_per_step": 1.2345678901234567,
             "per_unit": "u" * 60, "bytes": 1.2345678901234567e9} for m in range(40)]
    kernels = {f"kind{k}": {"ms_per_step": 1.2345678901234567, "launches_per_step": 8.0} for k in range(8)}
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}
    form = lambda: {"value": 9.7, "ms_per_step": 103.1, "kernels": kernels, "clocks": clocks, "per_level": rows,
                    "dloglik_per_obs_vs_fp64": 1.2345678901234567e-14}
    return {"metric": bench.METRIC, "value": 9.7, "unit": "evals/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 103.1, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": "w" * 40, "l2": "x" * 80},
            "roofline": {"bound": "tensor", "peak_source": "p" * 80, "per_level": rows, "kernels": kernels},
            "cpu_baseline": {"value": 0.19, "sample": "s" * 200, "oracle_check": {"regions": list(range(16))}},
            "e2e": {"value": 9.6, "unit": "evals/s", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 32},
            "gpu_launches": 640, "clocks": clocks, "emu": form(), "mixed": form(), "fp64": form(),
            "gradient": {"value": 3.1, "ms_per_step": 320.0, "fp64": form(), "mle": {"theta": [1.0] * 3}},
            "loglik": -1.0e6, "flops_per_step": 6.0e11, "batch": {"emu": {"ms_per_batch": 1071.4}, "datasets": 64},
            "prediction": {"emu": {"points_per_s": 1.0e7}, "grid": {"points": 1 << 20}}, "oracle_check": None,
            "level_J": {"ms_per_step": 110.0}}


def test_result_line_is_short_and_whole(capsys):
    line = full_line()
    bench.print_result(line)
    out = capsys.readouterr().out.splitlines()
    assert [l for l in out if l.startswith("{")] == out[-1:]
    assert len(out[-1]) < 4096
    short = json.loads(out[-1])
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert short[k] == line[k]
    assert short["batch_ms"] == {"emu": 1071.4} and short["prediction_points_per_s"] == {"emu": 1.0e7}
    tables = {l[len("# table "):].split(": ", 1)[0]: json.loads(l.split(": ", 1)[1]) for l in out[:-1]}
    assert tables["emu.per_level"] == line["emu"]["per_level"] and tables["batch"] == line["batch"]
    assert "per_level" in line["emu"] and line["oracle_check"] is None      # the argument is left as it was


def test_prediction_kernel_and_peak():
    fp64 = bench.prediction_kernel("fp64", 64, 0.86, 1700.0)
    assert (fp64["kernel"], fp64["pipe"], fp64["peak"]) == ("predict_kernel", "alu", bench.FP64_PEAK_TFLOPS)
    emu = bench.prediction_kernel("emu", 64, 3.9, 1700.0)
    assert (emu["kernel"], emu["pipe"], emu["peak"]) == ("predict_kernel_em", "tensor", 1700.0)
    assert emu["kernel_frac"] < 1.0
    assert bench.prediction_kernel("emu", 16, 0.5, 1700.0)["kernel"] == "predict_kernel"
