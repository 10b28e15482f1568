"""A context whose stream calls and captured step run different
implementations (a tuning cache can say so): each call continues from the last
forward, whichever ran it, and all agree with the oracle."""
import os

import numpy as np
import pytest
import torch

from oracle import dos_oracle as O
from paper_2604_02624_gb300 import _lib as L
from paper_2604_02624_gb300 import workloads as W
from paper_2604_02624_gb300.api import DiffractiveStack

from gpu_cases import TOL_FIELD, TOL_GRAD_ORACLE, TOL_LOSS, assert_close, oracle_model

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
DISP = np.array([[40e-9, -25e-9, 80e-9]])


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not os.path.exists(L.LIB_PATH):
        from paper_2604_02624_gb300 import build
        build.build()
    L.load()
    torch.cuda.set_device(DEV)


def _mixed(w, call, step, tmp_path, monkeypatch):
    """A context with the given choices, by way of a tuning cache."""
    cache = tmp_path / "tune"
    monkeypatch.setenv("DOS_TUNE_CACHE", str(cache))
    DiffractiveStack.from_workload(w, device=DEV).close()
    key = cache.read_text().splitlines()[0].split("\t")[0]
    cache.write_text(f"{key}\t{call}\t{step}\n")
    st = DiffractiveStack.from_workload(w, device=DEV)
    d = L.dos_describe(st.handle)
    assert d.startswith(f"path={call}") and f"step={step}" in d and "cache" in d, d
    return st


@pytest.mark.parametrize("call,step", [("fused:C4:L16", "multipass:bulk"), ("multipass", "fused:C2:L16"),
                                       ("multipass:bulk", "multipass")])
def test_calls_and_step_of_different_implementations(call, step, tmp_path, monkeypatch):
    w = W.workload("tiny")
    h = W.thickness(w, 0).astype(np.float32).astype(np.float64)
    T = W.targets(w, 1)
    st = _mixed(w, call, step, tmp_path, monkeypatch)
    path = st.path
    hd, Td = torch.tensor(h, dtype=torch.float32, device=DEV), torch.tensor(T, dtype=torch.float32, device=DEV)
    g = torch.empty_like(hd)

    def check(grad, disp, what):
        L_ref, _, ref, fwd = O.loss_and_grad(h, T, displacements=disp, **oracle_model(w))
        assert_close(grad.cpu().numpy().astype(np.float64), ref, TOL_GRAD_ORACLE, what)
        return L_ref, fwd

    for disp in (None, DISP, None):
        st.set_misalignment(disp)
        for again in range(2):  # capture, then replay
            val, _ = st.step(hd, Td, grad_out=g, read=True)
            L_ref, fwd = check(g, disp, "step")
            assert abs(val - L_ref) <= TOL_LOSS * L_ref
            assert_close(st.layer_field(1).cpu().numpy().astype(np.complex128), fwd["v"][:, 0], TOL_FIELD, "layer")
            _, _, dl = st.loss(Td)
            check(st.backward(dl), disp, "backward of the step")  # the step's fields and flags
            st.forward(hd)
            assert_close(st.layer_field(1).cpu().numpy().astype(np.complex128), fwd["v"][:, 0], TOL_FIELD, "layer")
            _, _, dl = st.loss(Td)
            check(st.backward(dl), disp, "forward, loss, backward")
            assert st.path == path
    st.close()


def test_step_keeps_the_thickness_for_a_later_backward():
    """The step's last kernel copies the thickness: a backward after the caller
    changed its buffer still uses the step's."""
    w = W.workload("tiny")
    h = W.thickness(w, 0).astype(np.float32).astype(np.float64)
    T = W.targets(w, 1)
    for path in ("multipass_bulk", "fused", "dft_gemm"):
        st = DiffractiveStack.from_workload(w, device=DEV, path=path)
        hd, Td = torch.tensor(h, dtype=torch.float32, device=DEV), torch.tensor(T, dtype=torch.float32, device=DEV)
        st.step(hd, Td)
        _, _, dl = st.loss(Td)
        hd.mul_(0.5)
        got = st.backward(dl).cpu().numpy().astype(np.float64)
        _, _, ref, _ = O.loss_and_grad(h, T, **oracle_model(w))
        assert_close(got, ref, TOL_GRAD_ORACLE)
        st.close()
