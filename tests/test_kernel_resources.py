"""Registers that the boundary kernels spill, as the compiler reports them: a
spilled word goes to local memory, for which the L1 has no room beside the
blocks' shared memory."""
import os
import re
import subprocess

import pytest

from paper_1307_0328_gb300 import build

# bytes of spill loads: a little above what the compiler reports (24, 0, 176
# and 128); with 940 the batched form ran slower than blocks of four warps
LIMIT = {"k_boundary": 64, "k_temporal": 64, "k_boundary_batch": 240, "k_temporal_batch": 240}


def test_boundary_kernels_spill_little():
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    cmd = [cc] + build.ARCH + build.FLAGS + ["-Xptxas", "-v", "-c", os.path.join(build.CSRC, "pmwa_kernels.cu"),
                                             "-o", os.devnull]
    log = subprocess.run(cmd, check=True, capture_output=True, text=True).stderr
    loads, name = {}, ""
    for line in log.splitlines():
        m = re.search(r"Compiling entry function '\w*?\d+(k_(?:boundary|temporal)(?:_batch)?)E", line)
        if "Compiling entry function" in line:
            name = m.group(1) if m else ""
        m = re.search(r"(\d+) bytes spill loads", line)
        if m and name:
            loads.setdefault(name, int(m.group(1)))  # (the kernel's own line comes first)
    assert set(loads) == set(LIMIT)
    assert all(loads[k] <= LIMIT[k] for k in LIMIT), loads
