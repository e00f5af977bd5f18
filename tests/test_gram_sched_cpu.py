"""The tile and K-share schedule of the tensor-core contraction
(gram_sched.cuh), checked on the host with the launcher's and the kernel's own
functions (tests/csrc/gram_sched_check.cu; no GPU): every entry in one tile,
every stage of a tile in one CTA, valid MMA shapes, no read past the buffer."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.skipif(shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"),
                    reason="needs nvcc")
def test_contraction_schedule(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = tmp_path / "gram_sched_check"
    subprocess.run([nvcc, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2406_01342_gb300", "csrc"),
                    "-I", os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "csrc", "gram_sched_check.cu"),
                    "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
