"""Subspace sizes of the FP64 Davidson: its projected eigenproblems (even and
odd dimensions, from one vector up to 24) against dense diagonalisation of the
library's own matrix elements <I|H|J> in the spin-flip-even sector.

Tolerance: a residual below r_tol = 1e-7 leaves an energy error of at most
r_tol^2 / gap, below 1e-10 for gaps above 1e-4 Eh.  1e-9 is asked for.
"""
import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from synth import make_chain

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("max_space", [4, 5, 11, 12, 13, 16, 17, 23, 24])
def test_lowest_state_with_every_subspace(max_space):
    chain = make_chain([3, 3, 2], 31)
    h1, eri = torch.tensor(chain.h, device=DEV), torch.tensor(chain.eri_packed(), device=DEV)
    with ifci.Handle(0, 0) as h:
        t = ifci.ifci_build_strings(h, 8, 3)
        nd = t.nstr ** 2
        I, J = torch.meshgrid(torch.arange(nd, device=DEV), torch.arange(nd, device=DEV), indexing="ij")
        H = ifci.ifci_h_elements(h, t, h1, eri, I.reshape(-1), J.reshape(-1)).cpu().numpy().reshape(nd, nd)
        e, _, st = ifci.ifci_davidson_batched(h, [ifci.CIProblem(8, 3, h1, eri, 0.0)] * 3,
                                              ifci.davidson_opts("fp64", r_tol=1e-7, max_space=max_space))
    a, b = np.triu_indices(t.nstr)
    S = np.zeros((nd, a.size))
    w = np.where(a == b, 0.5, np.sqrt(0.5))
    S[a * t.nstr + b, np.arange(a.size)] += w
    S[b * t.nstr + a, np.arange(a.size)] += w
    ref = np.linalg.eigvalsh(S.T @ H @ S)[0]
    assert list(st) == [0, 0, 0]
    assert np.abs(np.asarray(e) - ref).max() < 1e-9
