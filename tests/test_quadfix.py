"""The fixed-point quadrupole part of the FP64 form on the host (no GPU): its
terms and sums against long double, with the undefined-behaviour sanitizer."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fixed_point_quadrupole_terms(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    exe = str(tmp_path / "quadfix")
    cmd = [gxx, "-std=c++17", "-O1", "-ffp-contract=off", "-I" + os.path.join(ROOT, "paper_1206_1199_gb300", "csrc"),
           os.path.join(ROOT, "tests", "host_check", "quadfix.cpp"), "-o", exe]
    r = subprocess.run(cmd[:1] + ["-fsanitize=undefined"] + cmd[1:], capture_output=True, text=True)
    if r.returncode != 0 and "sanitize" in r.stderr:
        r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.stdout[-1000:], r.stderr[-2000:])
    assert "runtime error" not in r.stderr, r.stderr[-2000:]
