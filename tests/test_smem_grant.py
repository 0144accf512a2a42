"""Shared-memory grants are kept per device and hold under concurrent launches,
on CPU with a fake of the attribute call (tests/native/smem_grant.cpp); both
gather launchers use them."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1501_03869_gb300", "csrc")


def test_grants_per_device_and_thread(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not found")
    exe = str(tmp_path / "smem_grant")
    src = os.path.join(ROOT, "tests", "native", "smem_grant.cpp")
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-pthread", f"-I{CSRC}", src, "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout[-3000:]


def test_every_shared_memory_attribute_goes_through_a_grant():
    """The gathers' attribute call stands in one place, inside a grant (the
    bandwidth probe sets its own, one size, at every call)."""
    calls = []
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            calls += [name for line in f if "cudaFuncAttributeMaxDynamicSharedMemorySize" in line]
    assert calls == ["gather.cuh", "probe.cu"]
