"""No kernel has more static shared memory than the 48 KB that CUDA documents for
it (more is reached by dynamic shared memory after an opt-in): read from the
assembler's report on the kernels whose blocks hold the most."""
import os
import re
import subprocess

import pytest

from paper_2506_11273_gb300 import build as B


@pytest.mark.parametrize("unit", ["rr_keys.cu", "rr_trace.cu"])
def test_static_shared_memory(unit, tmp_path):
    out = subprocess.run([B._nvcc()] + B.ARCH + B.NVCC_FLAGS +
                         ["-Xptxas", "-v", "-c", os.path.join(B.CSRC, unit), "-o", str(tmp_path / "unit.o")],
                         capture_output=True, text=True, timeout=900)
    assert out.returncode == 0, out.stderr
    entry, used = None, {}
    for line in (out.stdout + out.stderr).splitlines():
        m = re.search(r"Compiling entry function '(\w+)'", line)
        entry = m.group(1) if m else entry
        m = re.search(r"Used \d+ registers.*?(\d+) bytes smem", line)
        if m:
            used[entry] = int(m.group(1))
    assert len(used) > 10
    assert not {k: v for k, v in used.items() if v > 48 * 1024}
