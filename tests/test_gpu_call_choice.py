"""The stream calls' implementation: the step's, unless fewer launches clearly
save the host time, and of the same number of launches the one whose kernels take
the least time, however the host's timing came out at create."""
import os
import re

import numpy as np
import pytest
import torch

from paper_2604_02624_gb300 import _lib as L
from paper_2604_02624_gb300.api import DiffractiveStack

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not os.path.exists(L.LIB_PATH):
        from paper_2604_02624_gb300 import build
        build.build()
    L.load()
    torch.cuda.set_device(DEV)


@pytest.mark.parametrize("n,m,k,nw", [(64, 128, 3, 16), (64, 128, 1, 4), (200, 400, 2, 6), (100, 200, 2, 8)])
def test_equal_launches_are_decided_by_the_kernels(n, m, k, nw):
    for _ in range(4):
        st = DiffractiveStack(n=n, m=m, n_layers=k, lambdas=np.linspace(480e-9, 720e-9, nw),
                              gaps=np.full(k + 1, 36e-6), pitch=300e-9, n_index=1.7, kappa=0.01, fov=n // 4 * 2, device=DEV)
        d = L.dos_describe(st.handle)
        ms = {c: float(v) for c, v in re.findall(r" (\S+)=([0-9.e+-]+)(?= |$)", d[d.index("(fwd+bwd ms):"):])}
        launch = ms.pop("launch")
        assert launch > 0
        ms = {re.sub(r"x\d+$", "", c): v for c, v in ms.items()}
        call = re.match(r"path=(\S+)", d).group(1)
        step = re.search(r" step=(\S+)", d.split("|")[0])
        step = step.group(1) if step else call
        assert ms[step] == min(ms.values())
        same = [v for c, v in ms.items() if c.startswith(call.split(":")[0])]  # all multi-pass or all cluster-resident
        assert ms[call] == min(same), d
        st.close()
