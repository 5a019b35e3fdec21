"""Long excitation lists of the fused FP64E sigma, around the limit of its narrow
epilogue (56 entries) and to the longest that small spaces have, against the
FP64 sigma; and integrals and vectors whose digits are all at their largest, so
that the level sums come close to the largest the digits allow.

Bound (that of the library's other FP64E sigma tests): 5e-10 of the norm and
5e-9 of max|sigma|.
"""
import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from synth import make_chain, random_ci_vector

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def close(h, t, h1, eri, c, sym):
    a = ifci.ifci_sigma(h, t, h1, eri, c, precision=ifci.IFCI_FP64E, spin_symmetric=sym).cpu().numpy()
    b = ifci.ifci_sigma(h, t, h1, eri, c, precision=ifci.IFCI_FP64).cpu().numpy()
    assert np.linalg.norm(a - b) <= 5e-10 * np.linalg.norm(b)
    assert np.max(np.abs(a - b)) <= 5e-9 * np.max(np.abs(b))


# lists of 54, 55, 56, 56 | 57, 60, 64, 68, 72, 76, 80, 84, 100 entries
@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("n,m", [(20, 3), (15, 5), (17, 14), (14, 7), (21, 3), (15, 6), (19, 16), (20, 17), (21, 18),
                                 (22, 19), (23, 20), (24, 21), (24, 20)])
def test_lists_at_the_limits_of_the_forms(n, m, sym):
    chain = make_chain([n // m + (1 if i < n % m else 0) for i in range(m)], 17 * n + m)
    h1, eri = torch.tensor(chain.h, device=DEV), torch.tensor(chain.eri_packed(), device=DEV)
    with ifci.Handle(0, 0) as h:
        t = ifci.ifci_build_strings(h, n, m)
        close(h, t, h1, eri, torch.tensor(random_ci_vector(t.nstr, t.nstr, seed=n + m, symmetric=sym), device=DEV), sym)


@pytest.mark.parametrize("n,m", [(17, 14), (21, 18), (23, 20)])
def test_largest_level_sums(n, m):
    # every digit of W and of c at its largest magnitude: x = 127.5 / 128 (1 + 2^-8 + ...)
    # has all its digits at +-128, in integrals and vector alike
    x = float(sum(127.5 / 128 * 2.0 ** (-8 * i) for i in range(5)))
    npair = n * (n + 1) // 2
    h1 = torch.zeros((n, n), dtype=torch.float64, device=DEV)
    eri = torch.full((npair, npair), 2 * x, dtype=torch.float64, device=DEV)
    with ifci.Handle(0, 0) as h:
        t = ifci.ifci_build_strings(h, n, m)
        c = torch.full((t.nstr, t.nstr), x, dtype=torch.float64, device=DEV)
        for sym in (True, False):
            close(h, t, h1, eri, c, sym)
