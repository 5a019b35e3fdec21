"""The FP64E sigma with every digit of W and of c near its largest and every
term of a string's contraction of one sign, so that the level accumulators and
the row sums come close to the bounds that the two forms of its epilogue rest
on: 2^22 a level in the narrow form (lists of up to 56 entries), 2^24 in the
wide one.

W is one number w = 2^-7 (127 + 127 2^-8 + ... + 127 2^-32) throughout (h1
cancels the exchange part of the fold exactly), |c| one number x, and the sign
of c[J][K] is s_J s_K, s_J the sign of the excitation I0 -> J of one string I0:
for alpha string I0 all contracted terms agree, and so do all beta terms of the
sum into S[I0][I0].  A host copy of the slicing checks the digits.

Tolerance: the products left out (digits i + j > 4) are at most 8 2^-40 of the
terms kept, the digits themselves are exact: 5e-10 of the norm and 5e-9 of
max|sigma|, the bound of the other FP64E sigma tests, against FP64.
"""
from fractions import Fraction

import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
NARROW = 56


def w_digits(w):
    r, out = Fraction(w) * 128, []   # scale 1: 1/2 <= |w| < 1
    for _ in range(5):
        out.append(round(r))         # to nearest, ties to even
        r = (r - out[-1]) * 256
    return out


def c_digits(x, dscale):
    v = round(Fraction(x) * 2 ** 38 / Fraction(dscale)) + 128 * 0x0101010101
    return [(v >> 8 * (4 - j) & (0x1FF if j == 0 else 0xFF)) - 128 for j in range(5)]


# lists of 42, 56, 56 | 60, 72, 100 entries
@pytest.mark.parametrize("n,m", [(16, 14), (17, 14), (14, 7), (22, 20), (21, 18), (24, 20)])
@pytest.mark.parametrize("sym", [True, False])
def test_levels_near_their_bounds(n, m, sym):
    ones = 127.0 * sum(2.0 ** (-8 * i) for i in range(5))
    w = ones / 128
    top = 31 if sym else 63             # |c| < dscale / 2 with spin-flip symmetry, < dscale without
    x = (top + (ones - 127.0)) / 64
    wd, cd = w_digits(w), c_digits(x, 1.0)   # both scales are 1
    assert wd == [127] * 5 and cd == [top] + [127] * 4
    K = m * (n - m + 1)
    level = max(K * sum(wd[i] * cd[L - i] for i in range(L + 1)) for L in range(5))
    if K == NARROW:
        assert 0.9 * 2 ** 22 < level < 2 ** 22
    assert level < 2 ** 24
    npair = n * (n + 1) // 2
    h1 = torch.full((n, n), n * w, dtype=torch.float64, device=DEV)   # = 1/2 sum_r (pr|rq): k_pq = 0
    eri = torch.full((npair, npair), 2 * w, dtype=torch.float64, device=DEV)
    with ifci.Handle(0, 0) as h:
        t = ifci.ifci_build_strings(h, n, m)
        I0 = t.nstr // 2
        row = t.exc.reshape(t.nstr, t.nexc)[I0].to(torch.int64)
        s = torch.ones(t.nstr, dtype=torch.float64, device=DEV)
        s[row >> 10] = 1.0 - 2.0 * (row & 1).to(torch.float64)
        c = x * s[:, None] * s[None, :]
        a = ifci.ifci_sigma(h, t, h1, eri, c.contiguous(), precision=ifci.IFCI_FP64E, spin_symmetric=sym)
        b = ifci.ifci_sigma(h, t, h1, eri, c.contiguous(), precision=ifci.IFCI_FP64)
        torch.cuda.synchronize()
    assert float((a - b).norm()) <= 5e-10 * float(b.norm())
    assert float((a - b).abs().max()) <= 5e-9 * float(b.abs().max())
