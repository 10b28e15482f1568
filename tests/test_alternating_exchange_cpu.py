"""The alternating exchange layouts of the line DFTs on the host: a round trip
through both layouts without the barrier between them, for every compiled line
shape and both pitches, and the bank mapping of the transposed T x T blocks in
the bulk column pass (8 lines x 4 element owners a warp)."""
import os
import shutil
import subprocess

import pytest

from test_bank_layout_cpu import BULK_COLUMN_M, SHAPES, ideal, wavefronts

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_NVCC = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
pytestmark = pytest.mark.skipif(_NVCC is None, reason="nvcc not available")


def test_round_trip_without_a_barrier(tmp_path):
    exe = str(tmp_path / "alternating")
    src = os.path.join(ROOT, "tests", "alternating_exchange_host.cu")
    p = subprocess.run([_NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-O1", "-x", "cu", src, "-o", exe],
                       capture_output=True, text=True)
    assert p.returncode == 0, p.stdout + p.stderr
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and "OK" in out.stdout, out.stdout


@pytest.mark.parametrize("m", BULK_COLUMN_M)
def test_transposed_blocks_are_conflict_free(m):
    """Entry (q = u + T j, k1) at row k1 + T j, column u: step 1 of owner t
    writes column t of each block (8 bytes), step 2 reads the rows t + T j in
    16-byte pairs."""
    c = SHAPES[m]
    Q, T, ZX, ZLB = c["Q"], c["T"], c["ZX"], c["ZLB"]
    for w in range(c["GT"] // 32):
        lanes = [((32 * w + i) % 8, (32 * w + i) // 8) for i in range(32)]  # (line, owner)
        for j in range(Q // T):
            for k1 in range(T):
                addrs = [lc * ZLB + (k1 + T * j) * ZX + t for lc, t in lanes]
                assert wavefronts(addrs, 1) == ideal(addrs, 1), (m, w, j, k1)
            for u in range(0, T, 2):
                addrs = [lc * ZLB + (t + T * j) * ZX + u for lc, t in lanes]
                assert wavefronts(addrs, 2) == ideal(addrs, 2), (m, w, j, u)
