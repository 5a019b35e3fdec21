"""The FP64E sigma scales its digits by powers of two of max|W| and max|c|:
multiplying the integrals or the vector by a power of two multiplies sigma by it
bit for bit, and zero stays zero.
"""
import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from synth import make_chain, random_ci_vector

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("n,m", [(3, 2), (9, 2), (12, 3)])
def test_sigma_scales_exactly(n, m, sym):
    chain = make_chain([n // m + (1 if i < n % m else 0) for i in range(m)], 7 * n + m)
    h1, eri = torch.tensor(chain.h, device=DEV), torch.tensor(chain.eri_packed(), device=DEV)
    with ifci.Handle(0, 0) as h:
        t = ifci.ifci_build_strings(h, n, m)
        c = torch.tensor(random_ci_vector(t.nstr, t.nstr, seed=n, symmetric=sym), device=DEV)

        def sigma(a, b):
            return ifci.ifci_sigma(h, t, h1 * 2.0 ** a, eri * 2.0 ** a, c * 2.0 ** b, precision=ifci.IFCI_FP64E,
                                   spin_symmetric=sym).cpu().numpy()

        ref = sigma(0, 0)
        assert np.abs(ref).max() > 0
        for a, b in [(1, 0), (0, -1), (30, -20), (-500, 300), (500, -300), (900, 0), (-900, 0), (0, 900), (0, -900)]:
            assert np.array_equal(sigma(a, b), ref * 2.0 ** (a + b)), (a, b)
        zero = [ifci.ifci_sigma(h, t, x * h1, x * eri, y * c, precision=ifci.IFCI_FP64E, spin_symmetric=sym)
                for x, y in ((0.0, 1.0), (1.0, 0.0), (0.0, 0.0))]
        assert all(not z.any().item() for z in zero)
