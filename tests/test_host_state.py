"""What the library's host threads share.  Contexts, batches and networks may be
driven from several threads at once, so every variable that outlives a call is
a once-flag, set under one, guarded by a mutex, or per thread."""
import glob
import os
import re
import subprocess

import pytest

# variable -> what makes it safe with several threads
SAFE = {"once": "std::once_flag", "fn": "set under tensor_map_encoder's once-flag", "g_scratch_mu": "the mutex itself",
        "g_scratch_ptr": "under g_scratch_mu", "g_noalloc_scratch": "under g_scratch_mu", "g_create_err[abi:cxx11]": "thread_local",
        "g_batch_create_err[abi:cxx11]": "thread_local", "g_net_err[abi:cxx11]": "thread_local"}


@pytest.fixture(scope="module")
def symbols():
    from paper_1805_07920_gb300 import _build, amh
    sources = glob.glob(os.path.join(_build.CSRC, "*")) + glob.glob(os.path.join(_build.INCLUDE, "*"))
    if not os.path.exists(amh.LIB_PATH) or os.path.getmtime(amh.LIB_PATH) < max(map(os.path.getmtime, sources)):
        _build.build()
    return subprocess.run(["nm", "-C", amh.LIB_PATH], capture_output=True, text=True, check=True).stdout.splitlines()


def test_no_unguarded_host_variables(symbols):
    found = set()
    for line in symbols:
        m = re.match(r"[0-9a-f]* [bBdD] (.*)", line)
        if not m or "amh" not in m[1] and "(anonymous namespace)" not in m[1]:
            continue
        if "guard variable" in m[1] or "__device_stub__" in m[1]:      # the compiler's kernel stubs
            continue
        found.add(m[1].split("::")[-1])
    assert "once" in found                                             # the listing works
    assert found <= set(SAFE), found - set(SAFE)
