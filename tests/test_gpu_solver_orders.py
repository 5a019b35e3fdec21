"""Both orders of the small eigenproblems in FP64E, at every P-space size from
one to 64 functions: an expansion keeps the serial order, a direct batch of the
same spaces takes the round-robin one, and FP64 decides.

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


@pytest.mark.parametrize("sizes", [(1, 2, 3, 4, 5), (6, 7, 8), (9, 10, 11), (2, 3, 3, 4), (5, 6, 2)])
def test_expansion_and_batch_reach_the_fp64_energies(sizes):
    chain = make_chain(list(sizes), 7 + len(sizes) + sizes[0])
    system = ifci.SystemArrays(chain.body_offsets, torch.tensor(chain.h, device=DEV),
                               torch.tensor(chain.eri_packed(), device=DEV))
    with ifci.Handle(0, 0) as h:
        ref = ifci.ifci_increments(h, system, 2, ifci.davidson_opts("fp64", r_tol=1e-7))
        out = ifci.ifci_increments(h, system, 2, ifci.davidson_opts("fp64e", r_tol=1e-7))
        assert np.all(out["status"] == 0)
        assert np.abs(out["e_x"] - ref["e_x"]).max() < 2e-9
        subs = ifci.body_subsets(len(sizes), 2)
        problems = []
        for X in subs:
            h1, eri, e_core = ifci.ifci_frozen_core(h, system, list(X))
            problems.append(ifci.CIProblem(sum(sizes[b] for b in X), len(X), h1, eri, e_core))
        e, _, st = ifci.ifci_davidson_batched(h, problems, ifci.davidson_opts("fp64e", r_tol=1e-7))
        assert np.all(np.asarray(st) == 0)
        assert np.abs(np.asarray(e) - ref["e_x"]).max() < 2e-9
