"""The smaller image that the w-plane transforms run on (resample_rule.cuh), checked on
the host with the plan's own rule and taps (tests/csrc/resample_rule_check.cu; no
GPU): the interpolation's error over the image and on its border, whatever share of the
turns the w-term has."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="needs nvcc")
def test_small_image_rule(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = tmp_path / "resample_rule_check"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2406_01342_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "csrc", "resample_rule_check.cu"), "-o", str(exe)],
                   check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
