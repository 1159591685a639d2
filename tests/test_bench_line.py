"""The benchmark prints one short line: the contract's keys whole, the tables on stderr (no GPU)."""
import importlib.util
import json
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_mod", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def full_line(bench):
    from paper_1204_0111_gb300 import workloads as wl
    table = {f"k_kernel_{i}": {"launches": 100 + i, "ms_per_step": 1.0 / 3, "tflops": 2.0 / 3, "gbs": 1e9 / 7} for i in range(30)}
    roof = {"kernel": "k_oz_gemm", "bound": "tensor", "achieved": 13.4 / 7, "peak": 54.1 / 3, "unit": "TFLOP/s", "frac": 0.25 / 3,
            "traffic": None, "kernel_share": 0.18 / 7, "timing": "x" * 120, "peak_source": "y" * 200}
    extra = {"workload": "z" * 300, "ms_per_step": 1e4 / 7, "gmres_iters": 11, "apply_ms": 464.0 / 3, "relres_max": 1e-6 / 3,
             "relres": 1e-6 / 3, "kernels": table, "roofline": roof, "sweep_tuning": table}
    return {"metric": bench.METRIC, "value": 0.94 / 7, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 1062.123456789, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": bench.config_dict(wl.cube_lens(100), 1, {"parallelism": "single GPU"}),
            "roofline": roof, "cpu_baseline": {"value": 0.0049, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 300},
            "e2e": {"value": 0.94 / 3, "unit": bench.UNIT, "steps": 5, "h2d_bytes_per_step": 24000000, "d2h_bytes_per_step": 16000000},
            "gpu_launches": 790, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}, "peaks": table,
            "rooflines": [roof] * 5, "detail": {"gmres_iters": 18, "relres": 1e-6 / 3, "apply_ms": 33.9, "setup_kernel_ms": 378.0,
                                                 "sweep_gbs": 1.0 / 3, "kernels": table, "sweep_tuning": table},
            "si_forms": table, "mixed": dict(extra, value=2.5 / 7), "salt256": extra, "layered200": extra, "batch16": extra}


def test_the_line_is_short_and_keeps_the_contract(bench):
    line = full_line(bench)
    out = bench.brief(line)
    assert len(json.dumps(out)) < 3000 < len(json.dumps(line))
    for k in bench.LINE_KEYS:
        assert k in out
    assert out["value"] == pytest.approx(line["value"], rel=1e-6) and out["e2e"]["h2d_bytes_per_step"] == 24000000
    assert out["config"] == json.loads(json.dumps(line["config"]))
    assert out["roofline"]["kernel"] == "k_oz_gemm" and "peak_source" not in out["roofline"]


def test_one_line_on_stdout_and_the_tables_on_stderr(bench, capsys):
    bench.report(full_line(bench))
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and "kernels" not in out
    assert "kernels" in json.loads(err)["detail"]
