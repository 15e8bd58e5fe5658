"""Host logic: the refinement residual in three FP32 words per number has no
more error than its FP64 form (flux_words_check.cpp, built with g++)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_residual_in_words_no_worse_than_fp64(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = tmp_path / "flux_words_check"
    subprocess.run([gxx, "-O2", "-std=gnu++17", "-ffp-contract=off", "-I", os.path.join(ROOT, "paper_1806_05619_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "flux_words_check.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
