"""Displaced layers on the column passes' own kernels: every compiled line
shape, with gaps that change length, shift sideways, do both or neither, and a
gap back to the aligned table; propagation of caller fields in both directions
over such gaps.  Against the FP64 oracle, at the FP32 paths' tolerances."""
import os

import numpy as np
import pytest
import torch

from oracle import dos_oracle as O
from paper_2604_02624_gb300 import _lib as L
from paper_2604_02624_gb300 import workloads as W
from paper_2604_02624_gb300.api import DiffractiveStack

from gpu_cases import TOL_FIELD, TOL_GRAD_ORACLE, assert_close, custom, oracle_model

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not os.path.exists(L.LIB_PATH):
        from paper_2604_02624_gb300 import build
        build.build()
    L.load()
    torch.cuda.set_device(DEV)


# three layers [pitch, pitch, wavelengths]: gap 0 shifts and changes, gap 1 only
# shifts, gap 2 only changes length, gap 3 does both; and all layers alike, where
# the gaps between them are the aligned ones
SHIFTS = {"mixed": [[1.3, -0.4, 0.2], [-2.1, 0.7, 0.2], [-2.1, 0.7, -0.6]], "alike": [[0.9, 1.1, 0.3]] * 3}


@pytest.mark.parametrize("path", ["multipass", "multipass_bulk"])
@pytest.mark.parametrize("kind", sorted(SHIFTS))
@pytest.mark.parametrize("n,m", [(8, 16), (13, 32), (32, 64), (64, 128), (100, 200), (101, 256), (40, 64), (200, 400)])
def test_displaced_gaps_match_oracle(n, m, kind, path):
    w = custom(n, m, 3, [480, 555, 690], 25, n - 2 * (n // 4), name="displaced")
    disp = np.array(SHIFTS[kind]) * np.array([w.pitch, w.pitch, w.lambda_mean])
    h = W.thickness(w, 0)
    hf = h.astype(np.float32).astype(np.float64)
    T = np.random.default_rng(m).uniform(0.0, 1.0, (3, w.fov, w.fov)).astype(np.float32)
    st = DiffractiveStack.from_workload(w, device=DEV, path=path)
    st.set_misalignment(disp)
    for _ in range(2):  # a second step builds the gaps' tables anew
        st.forward(torch.tensor(h, dtype=torch.float32, device=DEV))
        o = st.output_field().cpu().numpy().astype(np.complex128)
        _, _, dl = st.loss(torch.tensor(T, device=DEV))
        g = st.backward(dl).cpu().numpy().astype(np.float64)
    _, _, g_ref, fwd = O.loss_and_grad(hf, T.astype(np.float64), displacements=disp, **oracle_model(w))
    assert_close(o, fwd["o"], TOL_FIELD, "field")
    assert_close(g, g_ref, TOL_GRAD_ORACLE, "gradient")
    rng = np.random.default_rng(n)
    f = (rng.standard_normal((3, n, n)) + 1j * rng.standard_normal((3, n, n))).astype(np.complex64)
    for gap in range(4):
        for adj in (False, True):
            got = st.propagate(torch.tensor(f, device=DEV), gap, adj).cpu().numpy().astype(np.complex128)
            fn = O.propagate_adjoint if adj else O.propagate
            ref = np.stack([fn(f[i].astype(np.complex128), O.gap_transfer(w.lambdas[i], w.gaps, gap, m, w.pitch, 1.0,
                                                                         "decay", disp)) for i in range(3)])
            assert_close(got, ref, TOL_FIELD, (gap, adj))
    st.close()
