"""The reduction of the gradient parts over FP32's whole range: sums that leave it
on the way and come back, sums that stay outside, and a gradient written over the
thickness it belongs to."""
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


# one part per channel; 64 x 64 pixels in eight slices of the parts, 128 x 128 in one
@pytest.mark.parametrize("n,m,path", [(64, 128, "multipass"), (64, 128, "fused"), (128, 256, "multipass")])
def test_sums_outside_the_range(n, m, path):
    w = custom(n, m, 1, [600] * 6, 20, n // 2, name="range")  # six alike channels: six alike parts
    st = DiffractiveStack.from_workload(w, device=DEV, path=path)
    hd = torch.tensor(W.thickness(w, 0), dtype=torch.float32, device=DEV)
    st.forward(hd)
    seed = torch.zeros((6, w.fov, w.fov), device=DEV)
    seed[0] = torch.rand((w.fov, w.fov), generator=torch.Generator(DEV).manual_seed(1), device=DEV)
    one = st.backward(seed).cpu().numpy().astype(np.float64)  # a channel's part
    scale = float(np.float32(2.5e38 / np.abs(one).max()))
    for signs, total in (((1, 1, -1, 0, 0, 0), 1.0), ((1, 1, 1, -1, -1, -1), 0.0), ((1, 0, 0, 1, -1, 0), 1.0),
                         ((1, 1, 0, 0, 0, 0), 2.0), ((-1, -1, 0, -1, 0, 0), -3.0)):
        s = torch.stack([seed[0] * (scale * x) for x in signs])
        got = st.backward(s).cpu().numpy().astype(np.float64)
        want = one * scale * total
        inside = np.abs(want) < 3.3e38
        # FP32 fields of another scale: a part is the scaled one to rounding (1e-5 of the largest)
        assert np.all(np.isfinite(got[inside])) and np.max(np.abs(got - want)[inside]) <= 1e-5 * 2.5e38
        outside = np.abs(want) > 3.5e38
        assert np.array_equal(got[outside], np.sign(want[outside]) * np.inf)
        assert outside.any() == (abs(total) > 1.5)
    st.close()


@pytest.mark.parametrize("n,m", [(64, 128), (128, 256)])
def test_step_writes_its_gradient_over_the_thickness(n, m):
    w = custom(n, m, 1, [480, 555, 690], 20, n // 2, name="inplace")
    st = DiffractiveStack.from_workload(w, device=DEV, path="multipass_bulk")
    hd = torch.tensor(W.thickness(w, 0), dtype=torch.float32, device=DEV)
    T = torch.zeros((3, w.fov, w.fov), device=DEV)
    _, ref = st.step(hd, T)
    _, _, dl = st.loss(T, read=False)
    again = st.backward(dl).clone()
    for _ in range(3):
        x = hd.clone()
        st.step(x, T, grad_out=x)
        assert torch.equal(x, ref)
        _, _, dl = st.loss(T, read=False)
        assert torch.equal(st.backward(dl), again)  # with the thickness the step kept
    st.close()
