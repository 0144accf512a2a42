"""The nodes outside the mask, which every reconstruction clears, are listed in
runs of at most 512 that cover each of them once (tests/native/zero_runs.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1501_03869_gb300", "csrc")


def test_runs_are_short_and_cover_the_outside(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "zero_runs")
    cmd = [gxx, "-std=c++17", "-O1", "-pthread", f"-I{CSRC}", os.path.join(ROOT, "tests", "native", "zero_runs.cpp"),
           os.path.join(CSRC, "fmm_host.cpp"), os.path.join(CSRC, "const_host.cpp"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout[-2000:]
