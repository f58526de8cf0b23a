"""The arithmetic ceiling of bench.py reports the work that the kernels do."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_executed_instructions_are_those_of_the_row_kernels():
    src = open(os.path.join(ROOT, "paper_1004_3354_gb300", "csrc", "ed_internal.h")).read()
    body = re.search(r"void df_mac_row\(.*?\n}", src, re.S).group(0)
    n = len(re.findall(r"__f(?:add|sub|mul|maf)_rn\(", body))
    dim, nnz, ms = 41409225, 14.653, 0.58
    r = bench.alu_roofline("df64", dim, nnz, ms)["executed"]
    assert r["ops_per_launch"] == pytest.approx(dim * (nnz + 1.0) * n)
    assert r["frac"] == pytest.approx(dim * (nnz + 1.0) * n / (ms * 1e-3) / bench.FP32_PEAK, abs=1e-4)
    for prec in ("fp64", "fp32"):   # one instruction per multiply-add
        a = bench.alu_roofline(prec, dim, nnz, ms)
        assert a["executed"] == {"ops_per_launch": a["ops_per_launch"], "frac": a["frac"]}
