"""The fused FP64 sigma at the sizes where its loops can go wrong, against the
dense H of the library's own matrix elements <I|H|J> (checked element by element
elsewhere): one string, no empty or no occupied choice, odd counts of elements
and of excitations, several passes over the excitations, more strings than
threads; and, for larger spaces, against the FP64E sigma to that path's bound
(5e-10 of the norm).

Tolerance against the dense product: each element sums at most ~3000 products
of magnitudes below ~10, so rounding stays below 1e-12 of max|sigma|.
"""
import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from synth import make_chain, random_ci_vector

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def _space(h, n, m):
    chain = make_chain([n // m + (1 if i < n % m else 0) for i in range(m)], 57 * n + m)
    h1, eri = torch.tensor(chain.h, device=DEV), torch.tensor(chain.eri_packed(), device=DEV)
    t = ifci.ifci_build_strings(h, n, m)
    c = torch.tensor(random_ci_vector(t.nstr, t.nstr, seed=n + 3 * m), device=DEV)
    return h1, eri, t, c


@pytest.mark.parametrize("n,m", [(1, 1), (2, 1), (2, 2), (3, 2), (5, 1), (5, 4), (6, 3), (8, 4), (9, 2), (12, 2), (11, 1)])
def test_sigma64_equals_dense_h(n, m):
    with ifci.Handle(0, 0) as h:
        h1, eri, t, c = _space(h, n, m)
        s = ifci.ifci_sigma(h, t, h1, eri, c)
        nd = t.nstr ** 2
        I, J = torch.meshgrid(torch.arange(nd, device=DEV), torch.arange(nd, device=DEV), indexing="ij")
        H = ifci.ifci_h_elements(h, t, h1, eri, I.reshape(-1), J.reshape(-1)).reshape(nd, nd)
        torch.cuda.synchronize()
    ref = H @ c.reshape(-1)
    assert float((s.reshape(-1) - ref).abs().max()) <= 1e-12 * max(1.0, float(ref.abs().max()))


@pytest.mark.parametrize("n,m", [(13, 3), (10, 5), (18, 3), (12, 7), (14, 7), (31, 2)])
def test_sigma64_larger_spaces(n, m):
    with ifci.Handle(0, 0) as h:
        h1, eri, t, c = _space(h, n, m)
        s = ifci.ifci_sigma(h, t, h1, eri, c)
        again = ifci.ifci_sigma(h, t, h1, eri, c)
        if n <= 24:
            e = ifci.ifci_sigma(h, t, h1, eri, c, precision=ifci.IFCI_FP64E)
            assert float((s - e).norm()) <= 5e-10 * float(s.norm())
        else:   # too many pairs for the tensor-core path: the FP32 sigma, to its own bound
            e = ifci.ifci_sigma(h, t, h1, eri, c, precision=ifci.IFCI_FP32)
            assert float((s - e).abs().max()) <= 5e-5 * max(1.0, float(s.abs().max()))
        torch.cuda.synchronize()
    assert np.array_equal(s.cpu().numpy(), again.cpu().numpy())
