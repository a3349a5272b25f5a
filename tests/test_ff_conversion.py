"""The float-float of a double by integer instructions (ff.cuh) against the host's
IEEE conversions, at every exponent of its range and around it, ties included
(compiled as plain C++, no GPU)."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_integer_conversion_matches_ieee(tmp_path):
    exe = tmp_path / "ff_check"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math",
                        "-I", os.path.join(ROOT, "paper_1912_04457_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "ff_check.cpp"), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode != 0:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe), "3000000"], capture_output=True, text=True, timeout=300)
    cases, bad = map(int, r.stdout.split())
    assert cases == 3_000_000
    assert bad == 0 and r.returncode == 0
