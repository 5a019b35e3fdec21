"""The fused FP64E sigma at the sizes where its tiling can go wrong, against the
FP64 sigma: strings below, at and above the 128 of a tile; output pairs around
the chunks of 48 and their 16-wide remainders; excitation lists of one K step,
around 16, 32 and 48 rows, on both sides of the 51 where the accumulators stop
fitting 22 bits, and the longest that a small space has; with and without
spin-flip symmetry.

Bound (that of the library's other FP64E sigma tests): an element of the
contraction is off by at most npair (2^-38 + 2^-39) max|W| dscale, ~1e-9 of
max|W| dscale; 5e-10 of the norm and 5e-9 of max|sigma| are asked for.
"""
import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from synth import make_chain, random_ci_vector

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("n,m", [(1, 1), (2, 1), (3, 2), (5, 1), (5, 3), (6, 3), (9, 2), (9, 3), (16, 2), (17, 2), (10, 5),
                                 (18, 3), (19, 3), (20, 3), (13, 5), (24, 22), (23, 2), (12, 7)])
def test_fused_sigma_matches_fp64(n, m, sym):
    chain = make_chain([n // m + (1 if i < n % m else 0) for i in range(m)], 31 * n + m)
    h1, eri = torch.tensor(chain.h, device=DEV), torch.tensor(chain.eri_packed(), device=DEV)
    with ifci.Handle(0, 0) as h:
        t = ifci.ifci_build_strings(h, n, m)
        c = torch.tensor(random_ci_vector(t.nstr, t.nstr, seed=n + m, symmetric=sym), device=DEV)
        a = ifci.ifci_sigma(h, t, h1, eri, c, precision=ifci.IFCI_FP64E, spin_symmetric=sym)
        b = ifci.ifci_sigma(h, t, h1, eri, c, precision=ifci.IFCI_FP64)
        again = ifci.ifci_sigma(h, t, h1, eri, c, precision=ifci.IFCI_FP64E, spin_symmetric=sym)
        torch.cuda.synchronize()
    a, b = a.cpu().numpy(), b.cpu().numpy()
    assert np.array_equal(a, again.cpu().numpy())   # integer sums: the same in any order
    assert np.linalg.norm(a - b) <= 5e-10 * np.linalg.norm(b)
    assert np.max(np.abs(a - b)) <= 5e-9 * np.max(np.abs(b))
