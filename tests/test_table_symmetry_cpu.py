"""The quadrant tables are read transposed by the bulk column pass, so that the
bins' q = k^2 - fx^2 - fy^2 has to come out the same in either order.  The order
(k^2 - fx^2) - fy^2 does not, and neither does fx^2 + fy^2 with one square fused
into the addition; the sum of two rounded squares does."""
import os
import re
from fractions import Fraction

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2604_02624_gb300", "csrc")


def _bins():
    df = 1.0 / (512 * 300e-9)
    a = np.arange(258, dtype=np.float64) * df
    return (1.0 / 600e-9) ** 2, a[:, None], a[None, :]


def test_q_of_either_order():
    k2, fa, fb = _bins()
    assert np.array_equal(k2 - (fa * fa + fb * fb), k2 - (fb * fb + fa * fa))
    assert not np.array_equal(k2 - fa * fa - fb * fb, k2 - fb * fb - fa * fa)
    fused = lambda x, y: float(Fraction(x) ** 2 + Fraction(y * y))  # noqa: E731: fma(x, x, round(y y))
    col = [float(fa[i, 0]) for i in range(200, 240)]
    assert any(fused(x, y) != fused(y, x) for x in col for y in col)


def test_both_table_kernels_form_it_so():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "dos_setup.cu")).read())
    assert "__dsub_rn(k2, __dadd_rn(__dmul_rn(fa, fa), __dmul_rn(fb, fb)))" in src
    for kernel in ("k_htable", "k_sqtable"):
        body = src[src.index(f"__global__ void {kernel}("):]
        body = body[:body.index("cudaError_t launch")]
        assert "= bin_q(" in body and "fa * fa" not in body and "fb * fb" not in body
