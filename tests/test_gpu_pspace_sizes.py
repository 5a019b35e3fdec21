"""P-space sizes of the Davidson start: one to 64 pair functions (odd counts,
counts that are no multiple of four, the full 64 and spaces larger than it),
through both eigensolvers of the start (round-robin sweeps in an FP64 solve,
cyclic sweeps in an FP64E one), against dense diagonalisation of the library's
own matrix elements <I|H|J> in the spin-flip-even sector.

Tolerance: a residual below r_tol = 1e-7 leaves an energy error of at most
r_tol^2 / gap, below 1e-10 for gaps above 1e-4 Eh; the FP64E contraction adds
~1e-10 Eh.  2e-9 is asked for.
"""
import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from synth import make_chain

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("precision", ["fp64", "fp64e"])
@pytest.mark.parametrize("n,m", [(2, 1), (3, 1), (4, 1), (5, 1), (4, 2), (7, 1), (10, 1), (11, 1), (6, 2), (7, 3)])
def test_start_of_every_size_reaches_the_lowest_state(n, m, precision):
    chain = make_chain([n // m + (1 if i < n % m else 0) for i in range(m)], 100 * n + m)
    h1, eri = torch.tensor(chain.h, device=DEV), torch.tensor(chain.eri_packed(), device=DEV)
    with ifci.Handle(0, 0) as h:
        t = ifci.ifci_build_strings(h, n, m)
        nd = t.nstr ** 2
        I, J = torch.meshgrid(torch.arange(nd, device=DEV), torch.arange(nd, device=DEV), indexing="ij")
        H = ifci.ifci_h_elements(h, t, h1, eri, I.reshape(-1), J.reshape(-1)).cpu().numpy().reshape(nd, nd)
        e, _, st = ifci.ifci_davidson_batched(h, [ifci.CIProblem(n, m, h1, eri, 0.0)],
                                              ifci.davidson_opts(precision, r_tol=1e-7))
    a, b = np.triu_indices(t.nstr)
    S = np.zeros((nd, a.size))
    w = np.where(a == b, 0.5, np.sqrt(0.5))
    S[a * t.nstr + b, np.arange(a.size)] += w
    S[b * t.nstr + a, np.arange(a.size)] += w
    ref = np.linalg.eigvalsh(S.T @ H @ S)[0]
    assert st[0] == 0
    assert abs(e[0] - ref) < 2e-9
