"""FP64E Davidson batches in several sigma waves: a det_budget below the batch's
28 bytes per determinant splits it, down to one wave per problem, with short and
long excitation lists (narrow and wide epilogue) in one wave and apart, and with
sectored spaces.  Integer sums do not depend on the split: energies, iteration
counts and vectors are the same bit for bit.
"""
import math

import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from synth import chain_24_uneven, make_chain

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def _space(h, n, m, seed):
    chain = make_chain([n // m + (1 if i < n % m else 0) for i in range(m)], seed)
    return n, m, torch.tensor(chain.h, device=DEV), torch.tensor(chain.eri_packed(), device=DEV)


def _solve(h, spaces, budget):
    probs = [ifci.CIProblem(n, m, h1, eri, 0.0,
                            c_out=torch.empty(math.comb(n, m) ** 2, dtype=torch.float64, device=DEV))
             for n, m, h1, eri in spaces]
    before = h.launches()
    e, it, st = ifci.ifci_davidson_batched(h, probs, ifci.davidson_opts("fp64e", max_iter=40, det_budget=budget),
                                           allow_unconverged=True)
    torch.cuda.synchronize()
    return e, it, st, [p.c_out.cpu().numpy() for p in probs], h.launches() - before


# 6, 18, 60 (wide) and 42 entries a list; 1 element: one wave per problem
@pytest.mark.parametrize("budget", [1, 1 << 15, 250_000])
def test_waves_leave_the_result_unchanged(budget):
    with ifci.Handle(0, 0) as h:
        spaces = [_space(h, 4, 2, 1), _space(h, 22, 20, 2), _space(h, 8, 3, 3), _space(h, 22, 20, 4), _space(h, 16, 14, 5)]
        sysd_chain = chain_24_uneven()
        sysd = ifci.SystemArrays(sysd_chain.body_offsets, torch.tensor(sysd_chain.h, device=DEV),
                                 torch.tensor(sysd_chain.eri_packed(), device=DEV))
        for X in [(0, 12), (2, 20), (0, 1)]:   # far apart: blocks of decoupled bodies
            h1, eri, _ = ifci.ifci_frozen_core(h, sysd, X)
            spaces.append((h1.shape[0], len(X), h1, eri))
        # digit planes (2 x 5 FP16) and integer sums, in 8-byte elements: more than the budgets above
        need = [3.5 * math.comb(n, m) ** 2 for n, m, _, _ in spaces]
        assert sum(need) > 250_000
        one, many = _solve(h, spaces, 0), _solve(h, spaces, budget)
    assert many[4] > one[4]                    # more launches: it did run in waves
    for a, b in zip(one[:3], many[:3]):
        assert np.array_equal(a, b)
    for a, b in zip(one[3], many[3]):
        assert np.array_equal(a, b)
