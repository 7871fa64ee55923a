"""Sums of products in three floats stay within their derived bound and within
that of a sum in FP64 (CPU: the header is compiled for the host)."""
from __future__ import annotations

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_three_float_sum_is_finer_than_fp64(tmp_path):
    exe = tmp_path / "tf_sum"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off",
                           "-I", os.path.join(ROOT, "paper_2601_20569_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "cpp", "tf_sum.cpp"), "-o", str(exe)])
    v = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600,
                       check=True).stdout.split()
    assert float(v[1]) <= 1.0 and float(v[3]) <= 1.0, v
