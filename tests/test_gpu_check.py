"""An expired wait is reported to callers that read no loss: by dos_check after
propagation and after the last call of a program with an objective of its own,
and on the tensor-core paths by the next call as well.  The fault is made on the
host (DOS_INJECT_WAIT_TIMEOUT): a copy that is announced and never issued, or the
error flag itself."""
import os

import numpy as np
import pytest
import torch

from oracle import dos_oracle as O
from paper_2604_02624_gb300 import _lib as L
from paper_2604_02624_gb300 import workloads as W
from paper_2604_02624_gb300.api import DiffractiveStack, DosFunction

from gpu_cases import SPLIT_TARGET, TOL_FIELD, assert_close, oracle_model

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not os.path.exists(L.LIB_PATH):
        from paper_2604_02624_gb300 import build
        build.build()
    L.load()
    torch.cuda.set_device(DEV)


def _faulty(w, path, monkeypatch):
    monkeypatch.setenv("DOS_INJECT_WAIT_TIMEOUT", "1")
    st = DiffractiveStack.from_workload(w, device=DEV, path=path)
    monkeypatch.delenv("DOS_INJECT_WAIT_TIMEOUT")
    return st


def _reports(call):
    with pytest.raises(L.DosError) as e:
        call()
    return e.value.code == L.DOS_ERR_TIMEOUT


def test_propagation(monkeypatch):
    w = W.workload("tiny")
    st = _faulty(w, "multipass_bulk", monkeypatch)
    rng = np.random.default_rng(0)
    nw = len(w.lambdas)
    f = (rng.standard_normal((nw, w.n, w.n)) + 1j * rng.standard_normal((nw, w.n, w.n))).astype(np.complex64)
    fd = torch.tensor(f, device=DEV)
    st.propagate(fd, 0)  # gives up
    assert _reports(st.check)
    st.check()  # reported once
    got = st.propagate(fd, 0).cpu().numpy().astype(np.complex128)
    st.check()
    ref = np.stack([O.propagate(f[i].astype(np.complex128), O.gap_transfer(w.lambdas[i], w.gaps, 0, w.m, w.pitch, 1.0,
                                                                           "decay", None)) for i in range(nw)])
    assert_close(got, ref, TOL_FIELD)
    st.close()


@pytest.mark.parametrize("path", ["multipass_bulk", "dft_gemm"])
def test_own_objective(path, monkeypatch):
    w = W.workload("tiny")
    h = W.thickness(w, 0).astype(np.float32)
    st = _faulty(w, path, monkeypatch)
    hd = torch.tensor(h, device=DEV, requires_grad=True)
    I = DosFunction.apply(hd, st)  # gives up; nothing else is called
    torch.cuda.synchronize()
    assert _reports(st.check)
    I = DosFunction.apply(hd, st)
    torch.autograd.grad(I.sum(), hd)
    st.check()
    ref = O.forward(h.astype(np.float64), keep_fields=False, **oracle_model(w))["I"]
    assert_close(I.detach().cpu().numpy().astype(np.float64), ref, SPLIT_TARGET)
    st.close()


def test_the_next_tensor_core_call_reports(monkeypatch):
    w = W.workload("tiny")
    h = torch.tensor(W.thickness(w, 0), dtype=torch.float32, device=DEV)
    st = _faulty(w, "dft_gemm", monkeypatch)
    I = st.forward(h)
    torch.cuda.synchronize()
    assert _reports(lambda: st.backward(torch.ones_like(I)))  # before it queues anything
    I2 = st.forward(h)
    st.backward(torch.ones_like(I))
    st.check()
    assert torch.equal(I, I2)  # the flag alone was set
    st.close()
