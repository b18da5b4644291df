"""The update's launch arithmetic, checked on the host (launch_check.cpp), with the
shared memory the assembler reports for the kernels that state a carve-out."""
import os
import shutil
import subprocess

import pytest

from test_kernel_resources import _reports

HERE = os.path.dirname(os.path.abspath(__file__))


def test_launch_arithmetic(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    kernels = ("batch_phase_kernel", "batch_init_kernel", "12phase_kernel", "11init_kernel")     # one thread per pixel
    smem = {v["smem"] for k, v in _reports().items() if any(n in k for n in kernels) and v["smem"]}
    assert smem and min(smem) > 0
    exe = str(tmp_path / "launch_check")
    subprocess.run([gxx, "-std=c++17", "-O1", "-DSMEM=" + ",".join(map(str, sorted(smem))), "-o", exe,
                    os.path.join(HERE, "launch_check.cpp")], check=True, capture_output=True, timeout=120)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout[:2000] + r.stderr
    assert ", 0 failures" in r.stdout
