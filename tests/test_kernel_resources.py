"""What the assembler reports of the library's kernels."""
import glob
import os
import re

from paper_1805_07920_gb300 import _build, amh


def _reports():
    sources = glob.glob(os.path.join(_build.CSRC, "*")) + glob.glob(os.path.join(_build.INCLUDE, "*"))
    reports = [os.path.join(_build.OBJ_DIR, os.path.basename(s)[:-3] + ".ptxas") for s in _build.amh_sources()]
    if not all(map(os.path.exists, [amh.LIB_PATH, *reports])) or \
            min(map(os.path.getmtime, reports)) < max(map(os.path.getmtime, sources)):
        _build.build()
    out = {}
    for path in reports:
        name = None
        for line in open(path):
            m = re.search(r"Compiling entry function '(\w+)'", line)
            name = m[1] if m else name
            m = re.search(r"Used (\d+) registers.*", line)
            if m and name:
                smem = re.search(r"(\d+) bytes smem", line)
                out[name] = dict(registers=int(m[1]), smem=int(smem[1]) if smem else 0)
    return out


def test_static_shared_memory_within_48_kb():
    """More than 48 KB of shared memory has to be dynamic, with the opt-in; the
    toolkits do not promise more for static arrays."""
    kernels = _reports()
    assert len(kernels) > 60 and any("phase_kernel" in k for k in kernels)
    over = {k: v["smem"] for k, v in kernels.items() if v["smem"] > 48 * 1024}
    assert not over, over
