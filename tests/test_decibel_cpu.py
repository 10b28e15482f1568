"""The objective's decibels, on the host: half a unit in the last place is the
FP32 rounding of the result itself, which an FP64 logarithm would have as well;
0.05 more is allowed (the kernel's own error is bounded by 0.03)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_NVCC = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)


@pytest.mark.skipif(_NVCC is None, reason="nvcc not available")
def test_decibels_are_rounded_once(tmp_path):
    exe = str(tmp_path / "decibel")
    src = os.path.join(ROOT, "tests", "decibel_host.cu")
    p = subprocess.run([_NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-x", "cu", src, "-o", exe],
                       capture_output=True, text=True)
    assert p.returncode == 0, p.stdout + p.stderr
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout
