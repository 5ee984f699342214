"""The logarithm and circle of Box-Muller by table (csrc/tl_boxmuller.cuh) over the
uniforms of test_box_muller_header.py, in the roundings they cannot avoid."""
import os
import shutil
import subprocess

import pytest
from test_box_muller_header import MAIN, ROOT


def test_logarithm_and_circle_round_once_at_the_size_of_the_result(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "main.cpp", tmp_path / "bm"
    src.write_text(MAIN)
    subprocess.check_call([cxx, "-O2", "-std=gnu++17", "-I", os.path.join(ROOT, "paper_2607_24908_gb300", "csrc"),
                           str(src), "-o", str(exe)])
    log_worst, circle_worst = (float(v) for v in subprocess.check_output([str(exe)]).split()[:2])
    # the last sum, 2^-53 of the result; next to u = 1 the reduced argument and the polynomial,
    # half the result, another half each; a tenth for the rest
    assert log_worst <= 2.2 * 2.0 ** -53
    # half an ulp of a component below one, 2^-54; the product of the correction (0.0123) 2^-60
    assert circle_worst <= 1.05 * 2.0 ** -54
