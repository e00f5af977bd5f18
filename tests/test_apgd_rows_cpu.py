"""The rows of G that each CTA of the LASSO cluster takes (apgd_rows.cuh), checked on
the host with the kernel's own function (tests/csrc/apgd_rows_check.cu; no GPU): the
exchange of products relies on every CTA having some."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="needs nvcc")
def test_every_cta_has_rows(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = tmp_path / "apgd_rows_check"
    subprocess.run([nvcc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2406_01342_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "csrc", "apgd_rows_check.cu"), "-o", str(exe)],
                   check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
