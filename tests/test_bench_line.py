"""The line that `python bench.py` prints, made from the committed record of a run: short enough for a caller that keeps
the last 3000 characters of the output, with the output contract's keys and the record's own values (CPU)."""
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.fixture(scope="module")
def rec():
    with open(os.path.join(ROOT, "profiles", "bench_sweep.json")) as fh:
        return json.load(fh)


def test_line_fits_and_keeps_the_contract(rec):
    line = bench.short_line(rec)
    text = json.dumps(line)
    assert len(text) <= 2900 and "\n" not in text
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks"):
        assert line[k] == rec[k], k
    for k, names in (("e2e", ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")),
                     ("roofline", ("bound", "achieved", "peak", "unit", "frac", "traffic")),
                     ("cpu_baseline", ("value", "unit", "cores", "kind"))):
        assert all(line[k][n] == rec[k][n] for n in names), k


def test_every_leg_has_its_figure(rec):
    legs = bench.short_line(rec)["legs"]
    assert set(legs) == set(bench.LEG_FIGURES)
    assert legs["gemm_ms"] == pytest.approx(rec["gemm_bf16"]["ms"], rel=1e-4)


def test_a_run_without_a_cpu_baseline(rec):
    assert bench.short_line(dict(rec, cpu_baseline=None))["cpu_baseline"] is None
