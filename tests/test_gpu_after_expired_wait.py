"""Work queued after an expired wait, before the host has read the error: each
launch starts from its own items, so a forward that began after the failed one
is right although the flag is still to be reported."""
import os

import numpy as np
import pytest
import torch

from oracle import dos_oracle as O
from paper_2604_02624_gb300 import _lib as L
from paper_2604_02624_gb300 import workloads as W
from paper_2604_02624_gb300.api import DiffractiveStack

from gpu_cases import TOL_INTENSITY, assert_close, custom, oracle_model

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not os.path.exists(L.LIB_PATH):
        from paper_2604_02624_gb300 import build
        build.build()
    L.load()
    torch.cuda.set_device(DEV)


# channels: more items than resident blocks, so that the blocks draw from the counters
@pytest.mark.parametrize("force,inject", [("multipass:bulk[col]", "1"), ("multipass:bulk[col]", "2"),
                                          ("multipass:bulk[col]", "3"), ("multipass:bulk[row_fwd]", "1"),
                                          ("multipass:bulk[row_fwd]", "2")])
def test_forward_after_an_unread_expired_wait(monkeypatch, force, inject):
    nw = 6007
    w = custom(16, 32, 2, list(np.linspace(450, 740, nw)), 15, 10, name="draws")
    h = W.thickness(w, 0)
    monkeypatch.setenv("DOS_INJECT_WAIT_TIMEOUT", inject)
    monkeypatch.setenv("DOS_FORCE_CONFIG", force)
    st = DiffractiveStack.from_workload(w, device=DEV, path="auto")
    monkeypatch.delenv("DOS_INJECT_WAIT_TIMEOUT")
    monkeypatch.delenv("DOS_FORCE_CONFIG")
    assert force in L.dos_describe(st.handle)
    hd = torch.tensor(h, dtype=torch.float32, device=DEV)
    st.forward(hd)      # its first prefetching pass gives up
    I = st.forward(hd)  # nothing injected; the flag has not been read
    T = torch.zeros((nw, w.fov, w.fov), device=DEV)
    with pytest.raises(L.DosError) as e:
        st.loss(T)
    assert e.value.code == L.DOS_ERR_TIMEOUT
    ref = O.forward(h.astype(np.float32).astype(np.float64), keep_fields=False, **oracle_model(w))["I"]
    assert_close(I.cpu().numpy().astype(np.float64), ref, TOL_INTENSITY)
    st.close()
