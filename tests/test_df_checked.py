"""Strict mode's looper update in checked double-float arithmetic: wherever the
check accepts, the results are the FP64 update's bit for bit (CPU: the header is
compiled for the host), and it accepts all but a few of the fit's updates."""
from __future__ import annotations

import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_checked_update_is_the_fp64_update(tmp_path):
    exe = tmp_path / "df_checked"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off",
                           "-I", os.path.join(ROOT, "paper_2601_20569_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "cpp", "df_checked.cpp"), "-o", str(exe)])
    f = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600, check=True).stdout
    print(f)
    v = f.split()
    assert v[0] == "wrong" and int(v[1]) == 0
    # 20 results per update, each near a boundary with probability of about
    # 2^-18 times its cancellation (below 10 here): at least 99.9 % accepted
    assert float(v[3]) > 0.999
