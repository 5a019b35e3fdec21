"""ifci_davidson_expansion solves a batch as ifci_increments solves its body
sets: the same energies and iteration counts bit for bit, in the quantised and
mixed precisions and in FP64; and it is the call that the autotuner times."""
import numpy as np
import pytest
import torch

import paper_2307_10675_gb300 as ifci
from paper_2307_10675_gb300 import api, autotune
from synth import make_chain

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda", 0)
SIZES = (3, 4, 2, 5)


def _system():
    chain = make_chain(list(SIZES), 91)
    return ifci.SystemArrays(chain.body_offsets, torch.tensor(chain.h, device=DEV),
                             torch.tensor(chain.eri_packed(), device=DEV))


@pytest.mark.parametrize("precision", ["fp64", "fp64e", "bf16", "tf32"])
def test_batch_equals_the_expansion_bit_for_bit(precision):
    with ifci.Handle(0, 0) as h:
        system = _system()
        opts = ifci.davidson_opts(precision)
        out = ifci.ifci_increments(h, system, 3, opts)
        probs = []
        for X in ifci.body_subsets(len(SIZES), 3):
            h1, eri, e_core = ifci.ifci_frozen_core(h, system, list(X))
            probs.append(ifci.CIProblem(h1.shape[0], len(X), h1, eri, e_core))
        e, it, st = ifci.ifci_davidson_expansion(h, probs, opts)
    assert np.array_equal(e, out["e_x"])
    assert np.array_equal(it, out["iters"])
    assert np.all(st == 0)


def test_the_autotuner_times_it(monkeypatch):
    calls = []
    real = api.ifci_davidson_expansion

    def counted(*a, **k):
        calls.append(len(a[1]))
        return real(*a, **k)

    monkeypatch.setattr(api, "ifci_davidson_expansion", counted)
    with ifci.Handle(0, 0) as h:
        out = autotune.autotune(h, _system(), [(0, 1), (1, 2, 3)], "fp64e", grid={"max_space": [12, 8]})
    assert calls == [2] * (1 + len(out["table"]))


def test_a_set_by_itself():
    with ifci.Handle(0, 0) as h:
        system = _system()
        opts = ifci.davidson_opts("fp64e")
        out = ifci.ifci_increments(h, system, 2, opts)
        for i, X in enumerate(ifci.body_subsets(len(SIZES), 2)):
            h1, eri, e_core = ifci.ifci_frozen_core(h, system, list(X))
            e, _, _ = ifci.ifci_davidson_expansion(h, [ifci.CIProblem(h1.shape[0], len(X), h1, eri, e_core)], opts)
            assert e[0] == out["e_x"][i], X
