"""Bank mapping of the bulk column pass as its blocks run: one group of 8 columns,
thread = 8 t + line (owner t), every compiled size, M = 200 with its half-filled
last warp and its group astride the middle included.  The bank model and the
constants are test_bank_layout_cpu's."""
import pytest

from test_bank_layout_cpu import SHAPES, ideal, pytestmark, wavefronts  # noqa: F401

SIZES = sorted(SHAPES)


def _lanes(c, w):
    """(line, owner) of the lanes of warp w, None past the block's threads."""
    return [((32 * w + i) % 8, (32 * w + i) // 8) if 32 * w + i < c["GT"] else None for i in range(32)]


def _check(c, what, width, addr):
    for w in range((c["GT"] + 31) // 32):
        addrs = [addr(*x) if x else None for x in _lanes(c, w)]
        assert wavefronts(addrs, width) == ideal(addrs, width), (c["M"], what, w, addrs)


@pytest.mark.parametrize("m", SIZES)
def test_exchange_twiddles_and_stage(m):
    c = SHAPES[m]
    P, Q, T, ZX, ZLB, TWP = c["P"], c["Q"], c["T"], c["ZX"], c["ZLB"], c["TWP"]
    assert c["GT"] == 8 * T and c["GW"] == 8
    assert P == T, "the exchange layouts alternate"
    for j in range(Q // T):
        for k in range(0, P - 1, 2):
            _check(c, "row pairs", 2, lambda lc, t: lc * ZLB + (t + T * j) * ZX + k)
            _check(c, "twiddle pairs", 2, lambda lc, t: (t + T * j) * TWP + k)
        for k in range(P):
            _check(c, "transposed column", 1, lambda lc, t: lc * ZLB + (k + T * j) * ZX + t)
        for u in range(0, T - 1, 2):
            _check(c, "transposed row pairs", 2, lambda lc, t: lc * ZLB + (t + T * j) * ZX + u)
    for q in range(Q):
        _check(c, "column", 1, lambda lc, t: lc * ZLB + q * ZX + t)
    for i in range(m // T):
        _check(c, "stage", 1, lambda lc, t: (t + T * i) * 8 + lc)


@pytest.mark.parametrize("m", SIZES)
def test_transfer_table_tile(m):
    c = SHAPES[m]
    T, HP, HB = c["T"], c["HP"], c["HB"]
    for c0 in range(0, m, 8):
        row0 = c0 if c0 < m // 2 else m - c0 - 7
        hc = [min(c0 + lc, m - c0 - lc) - row0 for lc in range(8)]
        assert min(hc) >= 0 and max(hc) <= 7 and row0 >= 0
        for i in range(m // T):
            low = i < m // T // 2
            ky = lambda t: t + T * i if low else m - t - T * i  # noqa: B023,E731
            if c["STAGE_H"]:
                _check(c, ("tile", c0), 1, lambda lc, t: hc[lc] * HP + ky(t))
            else:
                box0 = T * i + T - 1 < HB if low else m - T * i < HB
                at = 0 if box0 else 8 * HB - (HP - HB)
                _check(c, ("tile", c0), 1, lambda lc, t: hc[lc] * HB + ky(t) + at)
