"""Rules by which batched launches choose their shapes, on CPU
(tests/native/row_rules.cpp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1501_03869_gb300", "csrc")


def test_rules(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "row_rules")
    src = os.path.join(ROOT, "tests", "native", "row_rules.cpp")
    r = subprocess.run([gxx, "-std=c++17", "-Wall", f"-I{CSRC}", src, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout[-3000:]
