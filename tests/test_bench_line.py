"""The benchmark's JSON line on the CPU: the contract's keys whole, the other
sections' main figures, and short enough for a reader that keeps a bounded tail
(a line of 20 KB was read as no line)."""
import importlib.util
import json
import os

import pytest

from tests.conftest import ROOT


@pytest.fixture(scope="module")
def bench():
    spec = importlib.util.spec_from_file_location("bench_under_test",
                                                  os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


def _record(bench, runs):
    stages = {"stage %d" % i: {"bytes_per_frame": 1.0 / 3, "ms_per_frame": 2.0 / 3,
                               "achieved_gbs": 1.1, "frac": 0.1} for i in range(9)}
    rec = {k: 1 for k in bench.CONTRACT_KEYS}
    rec.update(
        value=3411.3781872097884, ms_per_step=58.6,
        config={"workload": "w" * 200, "levels": 5},
        clocks={"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
        e2e={"value": 3374.25, "unit": "frames/s", "h2d_bytes_per_step": 653643504,
             "d2h_bytes_per_step": 1481932800, "call": "c" * 200},
        cpu_baseline={"value": 3.7, "sample": "s" * 200},
        path="p" * 400,
        in_order={"value": 2207.5, "call": "c" * 150},
        batched={"value": 4079.5, "stage_roofline": stages, "fp16_storage": {"value": 3988.0}},
        roofline={"frac": 0.093, "achieved": 634.1, "stage_roofline": stages,
                  "stage_share": {"s%d" % i: 0.1 for i in range(12)},
                  "kernel_io": {"kernel": "var_sor", "frac": 0.3}},
        serving={"runs": [{"p99_ms": 1.0 / 3, "by": stages}] * runs,
                 "sustainable": {"largest_rate_scale": 0.65}},
        multistream={"value": 12118.6, "autotune": {"346x260": {"candidates": [stages] * runs}}})
    return rec


@pytest.mark.parametrize("runs", [1, 6, 40])
def test_line_is_short_and_keeps_the_contract(bench, runs):
    rec = _record(bench, runs)
    line = bench.headline(rec)
    assert len(line) <= bench.LINE_LIMIT == 8000 and "\n" not in line
    out = json.loads(line)
    for k in bench.CONTRACT_KEYS:
        assert out[k] == rec[k], k
    assert out["roofline"]["frac"] == 0.093 and out["roofline"]["kernel_io"]["frac"] == 0.3
    assert out["in_order"]["value"] == 2207.5 and out["batched"]["value"] == 4079.5
    assert out["serving"]["sustainable"]["largest_rate_scale"] == 0.65
    assert out["multistream"]["value"] == 12118.6
    assert "runs" not in out["serving"]


def test_sections_go_before_the_contract_does(bench):
    rec = _record(bench, 2)
    for i in range(300):
        rec["extra %d" % i] = {"value": float(i), "note": "n" * 60}
    out = json.loads(bench.headline(rec))
    assert all(out[k] == rec[k] for k in bench.CONTRACT_KEYS) and "roofline" in out
    assert len(json.dumps(out)) <= bench.LINE_LIMIT


def test_kernel_io_counts_what_the_kernels_move(bench):
    """Against the sources: six coefficient planes, one flow and the four images
    of a coefficient launch, and 8 bytes of column words per 32 rows."""
    import re
    src = open(os.path.join(ROOT, "paper_2112_10591_gb300", "csrc", "k_var.cu")).read()
    names = re.search(r"enum \{ (kCI11[^}]*), kCPlanes \};", src).group(1)
    planes = len(names.split(","))
    geo = [(1280, 720, 318, 178), (640, 360, 158, 88)]
    P = 1280 * 720
    io = lambda s, l: bench.kernel_io_bytes_per_launch(s, l, geo, 275_000, P)
    assert io("var_coeff", 1) == (8 + 4 * 4 + 4 * planes) * 640 * 360
    assert io("var_sor", 0) == (4 * planes + 8 + 8) * P
    assert io("edt_cols", -1) == P + 8 * P / 32
    assert io("edt_rows_surface", -1) == 8 * P / 32 + 4 * P
    # the other stages have one layout
    for s, l in (("scatter", -1), ("patch_search", 0), ("densify", 1), ("flow_out", -1)):
        assert io(s, l) == bench.algorithmic_bytes_per_launch(s, l, geo, 275_000, P) > 0
