"""Memory of displaced designs: transfer tables are reserved for the gaps whose
length a displacement changes, when it first does, up to a number the caller may
set; every way to do with fewer gives the oracle's results."""
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


# three layers [pitch, pitch, wavelengths] and the gaps whose length changes
LATERAL = [[1.3, -0.4, 0.0], [-2.1, 0.7, 0.0], [0.4, 0.2, 0.0]], 0
ALIKE = [[0.9, 1.1, 0.3]] * 3, 2
ALL = [[1.3, -0.4, 0.2], [-2.1, 0.7, -0.3], [-2.1, 0.7, -0.6]], 4


@pytest.mark.parametrize("most", [None, 1, 0])
@pytest.mark.parametrize("n,m,path", [(40, 64, "multipass_bulk"), (64, 128, "multipass_bulk"), (64, 128, "multipass"),
                                      (13, 32, "multipass_bulk"), (64, 128, "fused")])
def test_tables_are_reserved_when_a_gap_changes_length(n, m, path, most, monkeypatch):
    if most is not None:
        monkeypatch.setenv("DOS_DISPLACED_TABLES", str(most))
    w = custom(n, m, 3, [480, 555, 690], 25, n - 2 * (n // 4), name="tables")
    h = W.thickness(w, 0)
    hf = h.astype(np.float32).astype(np.float64)
    T = np.random.default_rng(m).uniform(0.0, 1.0, (3, w.fov, w.fov)).astype(np.float32)
    st = DiffractiveStack.from_workload(w, device=DEV, path=path)
    quadrant = 3 * (m // 2 + 2) ** 2
    base = st.workspace_bytes
    held = 0
    g = torch.empty((3, n, n), device=DEV)
    for shifts, changed in (LATERAL, ALIKE, ALL, ALIKE, LATERAL):
        disp = np.array(shifts) * np.array([w.pitch, w.pitch, w.lambda_mean])
        st.set_misalignment(disp)
        if path.startswith("multipass"):
            most_kept = 4 if most is None else most
            held = max(held, changed if changed <= most_kept else min(1, most_kept))
        # the roots, and 8 bytes an entry for each table, 4 for the roots' remainders with the first
        assert st.workspace_bytes - base == quadrant * (4 + 8 * held + (4 if held else 0))
        _, _, ref, fwd = O.loss_and_grad(hf, T.astype(np.float64), displacements=disp, **oracle_model(w))
        hd, Td = torch.tensor(h, dtype=torch.float32, device=DEV), torch.tensor(T, device=DEV)
        for call in range(2):
            if call == 0:
                st.step(hd, Td, grad_out=g)
            else:
                st.forward(hd)
                _, _, dl = st.loss(Td)
                g = st.backward(dl)
            assert_close(st.output_field().cpu().numpy().astype(np.complex128), fwd["o"], TOL_FIELD, "field")
            assert_close(g.cpu().numpy().astype(np.float64), ref, TOL_GRAD_ORACLE, "gradient")
    st.close()
