"""The objective and gradient-reduction kernels at the edges of their ranges.

The objective is compared with its FP64 definition on the intensities that the
engine itself returned, so that only the kernel's own rounding is measured.
Tolerances: a thread sums at most (F_d^2 / 256 + 1) FP32 terms before FP64 takes
over, each term wrong by a few 2^-24 of its operands; with at most 20 terms the
sums are within 32 * 2^-24 = 2e-6 relative (1e-5 allowed), which moves a PSNR by
at most 10 / ln 10 * 1e-5 = 5e-5 dB; dL/dI is three roundings of the operands.
"""
import os

import numpy as np
import pytest
import torch

from oracle import dos_oracle as O
from paper_2604_02624_gb300 import _lib as L
from paper_2604_02624_gb300 import workloads as W
from paper_2604_02624_gb300.api import DiffractiveStack

from gpu_cases import TOL_GRAD_ORACLE, TOL_INTENSITY, assert_close, custom, oracle_model

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not os.path.exists(L.LIB_PATH):
        from paper_2604_02624_gb300 import build
        build.build()
    L.load()
    torch.cuda.set_device(DEV)


@pytest.mark.parametrize("loss", ["mse", "mse_scaled"])
@pytest.mark.parametrize("n,m,fov,b,nw", [
    (1, 16, 1, 1, 1),        # one detector pixel
    (20, 64, 16, 1, 3),      # exactly one pixel per thread
    (30, 64, 24, 3, 2),      # detector pixels of 3 x 3
    (64, 128, 64, 1, 300),   # 4096 detector pixels: the last size kept in shared memory
    (80, 200, 66, 1, 2),     # 4356: formed twice
    (140, 400, 132, 2, 2),   # 4356 detector pixels of 2 x 2
])
def test_objective_matches_its_definition(n, m, fov, b, nw, loss):
    w = custom(n, m, 1, list(np.linspace(480, 720, nw)), 20, fov, name="objective")
    st = DiffractiveStack.from_workload(w, device=DEV, path="multipass", loss=loss, detector_bin=b)
    rng = np.random.default_rng(fov * 10 + nw)
    T = rng.uniform(0.0, 1.0, (nw, fov // b, fov // b)).astype(np.float32)
    h = W.thickness(w, 0)
    I = st.forward(torch.tensor(h, dtype=torch.float32, device=DEV)).cpu().numpy().astype(np.float64)
    Td = torch.tensor(T, device=DEV)
    L_ref, p_ref, g_ref = O.mse_loss(I, T.astype(np.float64), scaled=(loss == "mse_scaled"), detector_bin=b)
    for _ in range(2):  # the second launch starts from the state the first one left
        val, psnr, g = st.loss(Td)
        assert abs(val - L_ref) <= 1e-5 * abs(L_ref) + 1e-12
        if fov > 1:  # one pixel: the scaled error is zero, its PSNR infinite or rounding
            assert np.max(np.abs(psnr.cpu().numpy() - p_ref)) <= 1e-4
        # one pixel: the scaled gradient is 2 sigma times a difference that vanishes
        scale = np.max(np.abs(g_ref)) if fov > 1 else 2.0 * max(1.0, float(T[0, 0, 0] / I[0, 0, 0]))
        assert np.max(np.abs(g.cpu().numpy() - g_ref)) <= 1e-5 * scale
    st.close()


@pytest.mark.parametrize("path,n,nw", [
    ("multipass", 13, 1), ("multipass", 13, 7), ("multipass", 13, 8), ("multipass", 13, 9), ("multipass", 13, 63),
    ("multipass", 13, 65), ("multipass", 13, 130),
    # the prefetching row passes, whose blocks draw chunks of channels: fewer channels than
    # resident blocks, a few per block, and many (ragged last chunks), even and odd rows
    ("multipass_bulk", 13, 1), ("multipass_bulk", 14, 5), ("multipass_bulk", 16, 700), ("multipass_bulk", 14, 3001),
    ("multipass_bulk", 13, 3001), ("multipass_bulk", 16, 6007),
])
def test_gradient_over_any_number_of_parts(path, n, nw):
    """Slices of the gradient parts that are empty, ragged, exactly one and more
    than one unrolled step long; chunks of one channel, of several, and cut short."""
    fov = n - 6
    w = custom(n, 32, 2, list(np.linspace(450, 740, nw)), 15, fov, name="parts")
    h = W.thickness(w, 0)
    T = np.random.default_rng(nw).uniform(0.0, 1.0, (nw, fov, fov)).astype(np.float32)
    st = DiffractiveStack.from_workload(w, device=DEV, path=path)
    hf = h.astype(np.float32).astype(np.float64)
    _, _, ref, fwd = O.loss_and_grad(hf, T.astype(np.float64), **oracle_model(w))
    for _ in range(2):  # the counters start from zero again
        I = st.forward(torch.tensor(h, dtype=torch.float32, device=DEV)).cpu().numpy().astype(np.float64)
        _, _, g = st.loss(torch.tensor(T, device=DEV))
        got = st.backward(g).cpu().numpy().astype(np.float64)
        assert_close(I, fwd["I"], TOL_INTENSITY)
        assert_close(got, ref, TOL_GRAD_ORACLE)
    st.close()
