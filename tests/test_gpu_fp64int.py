"""Sizes of the small eigensolvers and of the moment sums that their grouping
could get wrong: subspaces on both sides of the 16 that two problems share a
warp for, an odd number of problems in the batch, and moments of one to several
16 x 16 tiles (11 to 121 rows) against the gradient of the energy by central
differences of the library's own FP64 energies.

Davidson tolerance: residual 1e-8, error below 1e-14 / gap: 1e-9 asked for
between subspace sizes.  Differences: step 1e-4, truncation ~step^2 = 1e-8 of
the third derivative and rounding 1e-13 / 1e-4 = 1e-9: 1e-6 asked for.
"""
import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from synth import make_chain

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)


@pytest.mark.parametrize("precision", ["fp64", "fp64e"])
def test_subspace_sizes_agree(precision):
    probs = []
    for k, sizes in enumerate([[3, 2], [4, 3], [2, 2, 2], [5, 2], [3, 3, 2], [6], [2, 2]]):
        ch = make_chain(sizes, 900 + k)
        probs.append(ifci.CIProblem(sum(sizes), len(sizes), torch.tensor(ch.h, device=DEV),
                                    torch.tensor(ch.eri_packed(), device=DEV), 0.0))
    ref = None
    with ifci.Handle(0, 0) as h:
        for ms in (3, 12, 13, 16, 17, 24):
            e, _, st = ifci.ifci_davidson_batched(h, probs, ifci.davidson_opts(precision, max_space=ms, r_tol=1e-8,
                                                                               max_iter=400))
            assert np.all(st == 0)
            ref = e if ref is None else ref
            np.testing.assert_allclose(e, ref, rtol=0, atol=1e-9)


@pytest.mark.parametrize("sizes,order", [([4, 3], 1), ([5, 6], 2), ([3, 2, 3], 2), ([9, 6], 2), ([8, 7], 1)])
def test_gradient_tiles_match_differences(sizes, order):
    ch = make_chain(sizes, 40 + sum(sizes))
    V0 = ch.eri_packed()
    opts = ifci.davidson_opts("fp64", r_tol=1e-10, max_iter=300)
    rng = np.random.default_rng(5)
    with ifci.Handle(0, 0) as h:
        def system(hm, V):
            return ifci.SystemArrays(ch.body_offsets, torch.tensor(hm, device=DEV), torch.tensor(V, device=DEV))
        sysd = system(ch.h, V0)
        ifci.ifci_increments(h, sysd, order, opts)
        dh, dV = ifci.ifci_rdm_backward(h, sysd, order, 1.0, opts)
        dh, dV = dh.cpu().numpy(), dV.cpu().numpy()
        n = V0.shape[0]
        for _ in range(4):
            A, B = sorted(rng.integers(0, n, 2))
            e = []
            for step in (1e-4, -1e-4):
                V = V0.copy()
                V[A, B] += step
                if A != B:
                    V[B, A] += step
                e.append(ifci.ifci_increments(h, system(ch.h, V), order, opts)["e_total"])
            g = dV[A, B] + (dV[B, A] if A != B else 0.0)
            assert abs((e[0] - e[1]) / 2e-4 - g) < 1e-6
