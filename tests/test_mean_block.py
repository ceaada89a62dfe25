"""The float mean kernel's block test (csrc/prep.cu): a block of rows is added at
once, its sum of units onto the significand of s, when no value is a tie or too
large, no warp's total passes 2^53 and every running T of the block stays in
[2^52 + 1, 2^53 - 1]; or when, with 2^e above |s| + the sum of |x|, s and every
value are multiples of 2^(e - 53), so that no addition rounds.  Emulated in numpy against the index-order binary64 sum,
on the columns that exercise each branch of the 64-row step."""
from fractions import Fraction

import numpy as np
import pytest

from test_mean_scan import LO, HI, _bits, _columns, _double, _units


def block_sum(x, per, warp):
    """The sum with blocks of `per` rows, warps of `warp` rows, refused blocks
    added row by row; and how many blocks each rule took."""
    xb = x.view(np.uint32)
    s, accepted = 0.0, [0, 0]
    with np.errstate(over="ignore"):
        for b in range(0, x.size, per):
            c, cb = x[b:b + per], xb[b:b + per]
            sb = _bits(s)
            eb = (sb >> 52) & 0x7FF
            if eb not in (0, 0x7FF):
                S = (sb & ((1 << 52) - 1)) | (1 << 52)
                q, ok = _units(cb, eb - 1075, sb >> 63)
                q = [int(v) for v in q]
                totals = [sum(q[w:w + warp]) for w in range(0, len(q), warp)]
                T = S + np.cumsum(np.array(q, dtype=object))
                if ok.all() and all(abs(t) <= HI for t in totals) and LO <= min(T) and max(T) <= HI - 1:
                    s = _double((sb & ~((1 << 52) - 1)) | (int(T[-1]) - (1 << 52)))
                    accepted[0] += 1
                    continue
            top = np.float32((np.abs(c).astype(np.float32).sum(dtype=np.float32) + np.float32(abs(s))) * np.float32(1.001))
            if 0 < top < 1e30:
                g = int(np.frexp(top)[1]) - 53
                ms, es = int(sb & ((1 << 52) - 1)) | (1 << 52 if eb else 0), (eb or 1) - 1075
                sh = g - es
                assert sh >= 0
                ex = ((cb >> 23) & 0xFF).astype(np.int64)
                m = (cb & 0x7FFFFF).astype(np.int64) | np.where(ex != 0, 0x800000, 0)
                q = [Fraction(int(a)) * Fraction(2) ** (int(max(e, 1)) - 150 - g) for a, e in zip(m, ex)]
                if all(v.denominator == 1 for v in q) and ms % (1 << min(sh, 64)) == 0:
                    u = sum(int(-v if b >> 31 else v) for v, b in zip(q, cb)) + ((-1) ** (sb >> 63)) * (ms >> sh)
                    assert abs(u) < 1 << 53
                    s = float(np.ldexp(float(u), g))
                    accepted[1] += 1
                    continue
            for v in c:
                s = s + float(v)
    return s, accepted


@pytest.mark.parametrize("per,warp", [(2048, 256), (256, 256), (64, 32)])
def test_accepted_blocks_equal_the_index_order_sum(per, warp):
    columns = _columns()
    columns = columns.items() if isinstance(columns, dict) else columns
    taken = np.zeros(2, np.int64)
    for name, x in columns:
        x = np.ascontiguousarray(x, dtype=np.float32)
        ref = 0.0
        with np.errstate(over="ignore"):
            for v in x:
                ref = ref + float(v)
        got, accepted = block_sum(x, per, warp)
        assert _bits(got) == _bits(ref), name
        taken += accepted
    assert (taken > 0).all()  # both rules were met
