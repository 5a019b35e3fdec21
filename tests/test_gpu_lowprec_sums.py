"""Sums of the FP32 contraction (BF16, TF32, FP32 paths) in two floats, with one
and two tiles' buffers per SM (153 and 171 pairs), down to single strings.

Scaling the integrals by a power of two scales every product and partial sum
exactly while FP32 holds them: sigma follows bit for bit.  Where the scaled sums
leave FP32's range they are taken in FP64 instead; both ways are within 1e-13
of the exact sum of the same entries (2 x 48 additions of 2^-48), 1e-12 is asked
for.  The format's own error bounds the distance from FP64: 2^-8 (BF16), 2^-11
(TF32) or 2^-23 (FP32) per factor, two factors, at most twice that of the norm.
"""
import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from synth import make_chain, random_ci_vector

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("precision,eps", [("bf16", 2.0 ** -8), ("tf32", 2.0 ** -11), ("fp32", 2.0 ** -23)])
@pytest.mark.parametrize("n,m", [(2, 1), (3, 3), (5, 2), (12, 3), (16, 2), (17, 3), (18, 2)])
def test_scaled_sums(n, m, precision, eps):
    chain = make_chain([n // m + (1 if i < n % m else 0) for i in range(m)], 13 * n + m)
    h1, eri = torch.tensor(chain.h, device=DEV), torch.tensor(chain.eri_packed(), device=DEV)
    with ifci.Handle(0, 0) as h:
        t = ifci.ifci_build_strings(h, n, m)
        for sym in (True, False):
            c = torch.tensor(random_ci_vector(t.nstr, t.nstr, seed=n * m, symmetric=sym), device=DEV)

            def sigma(k, prec=ifci.PRECISIONS[precision]):
                return ifci.ifci_sigma(h, t, h1 * 2.0 ** k, eri * 2.0 ** k, c, precision=prec, spin_symmetric=sym).cpu().numpy()

            ref, exact = sigma(0), sigma(0, ifci.IFCI_FP64)
            assert np.linalg.norm(ref - exact) <= 4 * eps * np.linalg.norm(exact)
            assert np.array_equal(sigma(20), ref * 2.0 ** 20)
            # H = 2 m on the whole space, as 2 m equal terms per determinant: with the
            # vector near FP32's largest number the terms fit and their sums do not
            one, none = torch.eye(n, device=DEV, dtype=torch.float64), torch.zeros_like(eri)

            def number(k):
                return ifci.ifci_sigma(h, t, one, none, c * 2.0 ** k, precision=ifci.PRECISIONS[precision],
                                       spin_symmetric=sym).cpu().numpy()

            k = 126 - int(np.floor(np.log2(c.abs().max().item())))
            ref, big = number(0), number(k)
            assert np.isfinite(big).all()
            assert np.abs(big - ref * 2.0 ** k).max() <= 1e-12 * np.abs(big).max()
