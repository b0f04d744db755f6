"""The integer-pipe double-precision multiply, divide and square root of the FP64
tracer (csrc/soft64.cuh), compiled for the host and compared bit for bit with
the processor's operations (tests/soft64_check.cu). No GPU is used."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_integer_operations_round_as_the_processor_does(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "soft64_check")
    src = os.path.join(ROOT, "tests", "soft64_check.cu")
    inc = os.path.join(ROOT, "paper_2208_12569_gb300", "csrc")
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off", "-I", inc, src, "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe, "5000000"], capture_output=True, text=True, timeout=300)
    n, bad = (int(v) for v in out.stdout.split("\n")[-2].split())
    assert out.returncode == 0 and bad == 0 and n > 30_000_000, out.stdout
