"""Backward pass over a set of 3.3e6 determinants, whose moments are summed in
more than the fewest determinants per chunk: the partial sums of a wave stay
below 64 jobs of 32 KB per SM (and one a problem), next to the gathered rows of
the largest set, and the gradient keeps Euler's identity.

Tolerance: E is homogeneous of degree one in (h, V) and the gradient is taken at
vectors converged to r_tol = 1e-7, whose energies are off by r_tol^2 / gap
~1e-13; FP64E energies and FP64 moments differ by ~1e-9 Eh.  1e-8 is asked for.
"""
import math

import pytest
import torch

import paper_2307_10675_gb300 as ifci
from synth import make_chain

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


def test_partial_sums_are_bounded():
    chain = make_chain([4, 4, 4, 4], 44)
    h1, V = torch.tensor(chain.h, device=DEV), torch.tensor(chain.eri_packed(), device=DEV)
    system = ifci.SystemArrays(chain.body_offsets, h1, V)
    opts = ifci.davidson_opts("fp64e", r_tol=1e-7, max_iter=300)
    with ifci.Handle(0, 0) as h:
        out = ifci.ifci_increments(h, system, 4, opts)
        before = h.workspace_bytes()
        dh, dV = ifci.ifci_rdm_backward(h, system, 4, 1.0, opts)
        torch.cuda.synchronize()
        grown = h.workspace_bytes() - before
    rows = 8 * (16 * 17 // 2 + 1) * math.comb(16, 4) ** 2
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # tables, work lists and moments take less than 64 MB; the workspace grows an eighth beyond the need
    assert grown <= 1.125 * (rows + 32768 * (64 * sms + 64) + (64 << 20))
    euler = float((h1 * dh).sum() + (V * dV).sum())
    assert abs(euler - out["e_total"]) <= 1e-8
