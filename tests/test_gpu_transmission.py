"""The transmission of Eq. 1 over any thickness: phases of thousands of cycles of
either sign, quarter turns, zero and values below FP32's normal range.

With every gap zero and a full aperture the output field is t(h) itself, through
two FP32 DFT pairs.  Their rounding, ~3e-7 of the field's root mean square (1),
dominates; 2e-6 absolute is six times that at every element.  The reference takes
the same float thickness and FP64 constants."""
import os

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


@pytest.mark.parametrize("scale", [0.0, 1e-42, 1e-9, 1e-6, 1e-4, 5e-3, "quarters"])
@pytest.mark.parametrize("path", ["multipass", "multipass_bulk"])
def test_transmission_over_any_thickness(path, scale):
    n, lam = 32, np.array([450e-9, 612.5e-9, 750e-9])
    idx, base = np.array([1.7, 1.52, 1.33]), 120e-9
    rng = np.random.default_rng(7)
    if scale == "quarters":  # multiples of an eighth of a turn of the first channel
        h = (np.arange(n * n) - n * n // 2).reshape(1, n, n) * (lam[0] / (idx[0] - 1.0) / 8.0)
    else:
        h = rng.uniform(-1.0, 1.0, (1, n, n)) * scale
    h32 = h.astype(np.float32)
    st = DiffractiveStack(n=n, m=64, n_layers=1, lambdas=lam, gaps=[0.0, 0.0], pitch=300e-9, n_index=idx, kappa=0.0,
                          fov=n, h_base=base, path=path, device=DEV)
    st.forward(torch.tensor(h32, device=DEV))
    got = st.output_field().cpu().numpy()
    cycles = ((idx - 1.0) / lam)[:, None, None] * (h32.astype(np.float64) + base)
    # an FP32 phase constant is an FP32 pair: 2^-48 of the phase, below 1e-9 cycles here
    ref = np.exp(-2j * np.pi * (cycles - np.rint(cycles)))
    assert np.max(np.abs(got - ref)) <= 2e-6
    st.close()
