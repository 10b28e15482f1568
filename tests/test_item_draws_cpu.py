"""The counter that the prefetching passes draw their items from, on the host."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_NVCC = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)


@pytest.mark.skipif(_NVCC is None, reason="nvcc not available")
def test_counter_is_zero_after_every_launch(tmp_path):
    exe = str(tmp_path / "draws")
    src = os.path.join(ROOT, "tests", "item_draws_host.cu")
    p = subprocess.run([_NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-x", "cu", src, "-o", exe],
                       capture_output=True, text=True)
    assert p.returncode == 0, p.stdout + p.stderr
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and "OK" in out.stdout, out.stdout
