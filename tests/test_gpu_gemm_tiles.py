"""The GEMM path on tiles of 128 and of 256 columns.

Few tiles take narrow columns, many wide ones; a launch's columns may end in the
first or the second half of a stored 256-row operand tile, or fill it.  Against
the FP64 oracle: each GEMM of two-part operands adds about 1.1e-5 (relative L2)
to the field, 12 of them to the output and 20 to the gradient's two fields, so
8e-5 is expected of the intensity and 1e-4 of the gradient with a seed of the
difference I - T; five times that is allowed.  A wrong or missing half tile is
wrong by tens of percent.
"""
import os

import numpy as np
import pytest
import torch

from oracle import dos_oracle as O
from paper_2604_02624_gb300 import _lib as L
from paper_2604_02624_gb300 import workloads as W
from paper_2604_02624_gb300.api import DiffractiveStack

from gpu_cases import assert_close, custom, oracle_model

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not os.path.exists(L.LIB_PATH):
        from paper_2604_02624_gb300 import build
        build.build()
    L.load()
    torch.cuda.set_device(DEV)


@pytest.mark.parametrize("path", ["dft_gemm", "dft_gemm_x3"])
@pytest.mark.parametrize("n,m,nw", [
    (6, 16, 1),     # all columns in half a tile
    (64, 128, 2),   # exactly half a tile, exactly one
    (64, 128, 3),   # one and a half
    (101, 256, 7),  # ragged: 707 columns
    (200, 400, 1),  # 200 and 800 columns
    (60, 200, 90),  # many tiles: wide, the narrow ones a wave more
])
def test_narrow_and_wide_tiles(path, n, m, nw):
    fov = n // 2 - (n - n // 2) % 2
    w = custom(n, m, 2, list(np.linspace(480, 720, nw)), 25, fov, name="tiles")
    h = W.thickness(w, 0)
    T = np.random.default_rng(n + nw).uniform(0.0, 1.0, (nw, fov, fov)).astype(np.float32)
    _, _, ref, fwd = O.loss_and_grad(h.astype(np.float32).astype(np.float64), T.astype(np.float64), **oracle_model(w))
    st = DiffractiveStack.from_workload(w, device=DEV, path=path)
    I = st.forward(torch.tensor(h, dtype=torch.float32, device=DEV)).cpu().numpy().astype(np.float64)
    _, _, g = st.loss(torch.tensor(T, device=DEV))
    got = st.backward(g).cpu().numpy().astype(np.float64)
    assert_close(I, fwd["I"], 5e-4)
    assert_close(got, ref, 5e-4)
    st.close()
