"""The objective's sums do not depend on the block that forms them.

A sum is 256 FP32 partials, added two by two as FP32 pairs and then in FP64:
partial i holds the pixels i, i + 256, ... as a chain of FP32
multiply-adds.  The same is formed here, in NumPy, from the
intensities that the engine returned: each multiply-add exactly (the product of
two FP32 numbers is exact in FP64, and the FP64 sum with an FP32 number is rounded
once more to FP32; at most one in 2^29 of those is rounded twice).  The loss and
the PSNR, FP64 quotients of the sums, then agree to FP64 rounding and to FP32's."""
import os

import numpy as np
import pytest
import torch

from paper_2604_02624_gb300 import _lib as L
from paper_2604_02624_gb300 import workloads as W
from paper_2604_02624_gb300.api import DiffractiveStack

from gpu_cases import custom

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not os.path.exists(L.LIB_PATH):
        from paper_2604_02624_gb300 import build
        build.build()
    L.load()
    torch.cuda.set_device(DEV)


def _sum(a, b):
    """Sum over the pixels of a b, [channels][pixels] float32, as 256 FP32 chains."""
    nw, px = a.shape
    pad = -px % 256
    a, b = (np.pad(x, ((0, 0), (0, pad))).reshape(nw, -1, 256) for x in (a, b))
    acc = np.zeros((nw, 256), np.float32)
    for i in range(a.shape[1]):
        acc = (a[:, i].astype(np.float64) * b[:, i].astype(np.float64) + acc.astype(np.float64)).astype(np.float32)
    return acc.astype(np.float64).sum(1)


# side of the output plane: fewer pixels than 128, than 256, a second stride cut
# short, the largest that takes the small block and the first that does not
@pytest.mark.parametrize("loss", ["mse", "mse_scaled"])
@pytest.mark.parametrize("fov", [6, 14, 20, 34, 36])
@pytest.mark.parametrize("nw", [200, 1025])  # above 1024 channels: the small block
def test_sums_are_256_chains(fov, loss, nw):
    w = custom(40, 128, 1, list(np.linspace(450, 740, nw)), 20, fov, name="chains")
    st = DiffractiveStack.from_workload(w, device=DEV, path="multipass", loss=loss)
    T = np.random.default_rng(fov).uniform(0.0, 1.0, (nw, fov, fov)).astype(np.float32)
    I = st.forward(torch.tensor(W.thickness(w, 0), dtype=torch.float32, device=DEV)).cpu().numpy()
    val, psnr, _ = st.loss(torch.tensor(T, device=DEV))
    I, T = I.reshape(nw, -1), T.reshape(nw, -1)
    d = I - T
    sg = (_sum(I, T) / _sum(I, I)).astype(np.float32)[:, None]
    ds = (sg.astype(np.float64) * I.astype(np.float64) - T.astype(np.float64)).astype(np.float32)
    ssc = _sum(ds, ds)
    want = (ssc if loss == "mse_scaled" else _sum(d, d)).sum() / (nw * fov * fov)
    assert abs(val - want) <= 1e-12 * want
    p = 10.0 * np.log10(fov * fov / ssc)
    # half a unit in the last place of the result, and the kernel's 0.03 before it
    assert np.max(np.abs(psnr.cpu().numpy().astype(np.float64) - p) / np.spacing(np.abs(p).astype(np.float32))) <= 0.55
    st.close()


def test_sums_past_the_single_precision_range():
    """Targets so large that two of a sum's FP32 partials leave FP32's range
    together though neither does: the loss is the FP64 sum."""
    w = custom(40, 128, 1, [600], 20, 20, name="range")
    st = DiffractiveStack.from_workload(w, device=DEV, path="multipass")
    st.forward(torch.tensor(W.thickness(w, 0), dtype=torch.float32, device=DEV))
    T = np.full((1, 20, 20), 1.5e19, np.float32)  # (I - T)^2 = 2.25e38, 400 of them in 256 partials
    T[0, 0, 256 % 20:] = 1.0
    T = T.reshape(-1)
    T[256:] = 1.0  # one large term a partial at most
    val, _, _ = st.loss(torch.tensor(T.reshape(1, 20, 20), device=DEV), psnr=False, grad=False)
    want = np.count_nonzero(T > 2.0) * float(np.float32(1.5e19)) ** 2 / 400.0
    assert np.isfinite(val) and abs(val - want) <= 1e-6 * want
    st.close()
