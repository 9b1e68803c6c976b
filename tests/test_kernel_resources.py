"""What the compiler reports of the small kernels' static shared memory: 48 KB is what CUDA
documents for it on every device."""
import os
import re
import subprocess

import pytest

from paper_2106_08040_gb300 import build


def static_shared_bytes(source, tmp_path):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    cmd = [nvcc] + build.ARCH + ["-O3", "-std=c++17", "-Xptxas", "-v", "-I",
                                 os.path.join(build.HERE, "..", "include"), "-cubin",
                                 os.path.join(build.CSRC, source), "-o", str(tmp_path / "out.cubin")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    used = [re.search(r"(\d+) bytes smem", line) for line in r.stderr.splitlines() if "Used " in line]
    assert used
    return [int(m.group(1)) if m else 0 for m in used]


@pytest.mark.parametrize("source", ["fp_models.cu", "fp_m2.cu"])
def test_static_shared_memory_is_within_48_kb(source, tmp_path):
    assert max(static_shared_bytes(source, tmp_path)) <= 48 * 1024
