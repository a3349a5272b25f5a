"""The integer binary64 product, quotient and square root (exact64.cuh) against the host's IEEE
operations, bit for bit, with FP32 estimates off by up to two units in the last place
(compiled as plain C++, no GPU)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_integer_division_and_root_match_ieee(tmp_path):
    exe = tmp_path / "div64_check"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math",
                        "-I", os.path.join(ROOT, "paper_1912_04457_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "div64_check.cpp"), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe), "10000000"], capture_output=True, text=True, timeout=300)
    cases, bad = map(int, r.stdout.split())
    assert cases == 30_000_000
    assert bad == 0 and r.returncode == 0
