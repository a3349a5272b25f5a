"""Every momentum grid takes the mirrored forms of the drift and the moments, those whose
central cell is not exactly 0 in FP32 among them (compiled as plain C++, no GPU)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_grid_is_mirrored(tmp_path):
    exe = tmp_path / "octet_check"
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(cuda, "include"),
                        "-I", os.path.join(ROOT, "paper_1912_04457_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "octet_check.cpp"), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    cases, off, bad = map(int, r.stdout.split())
    assert cases == 256 * 40 and off > 0
    assert bad == 0 and r.returncode == 0
