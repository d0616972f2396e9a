"""The key quantisation's FP32 evaluation (csrc/keys_quant.cuh) equals the FP64 expression wherever it decides,
checked on the host on ~5e6 operands."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1610_07279_gb300", "csrc")


def test_fp32_quantisation_matches_fp64(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "keys_quant_fp32_check")
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-I", CSRC, os.path.join(HERE, "keys_quant_fp32_check.cpp"),
                    "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    w = r.stdout.split()
    cases, decided, bad = int(w[1]), int(w[3]), int(w[5])
    assert bad == 0 and decided > cases // 3, r.stdout  # random positions are decided but for 1 in 2^18
