"""bench.paths_sample reports the solver that an expansion runs (no GPU: the
library is a stand-in that records the calls)."""
import os
import sys
from types import SimpleNamespace

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
from synth import chain_24_uneven  # noqa: E402


def test_paths_sample_solves_as_an_expansion():
    calls = []

    def solve(handle, probs, opts, allow_unconverged=False):
        calls.append(opts["precision"])
        n = len(probs)
        return np.zeros(n), np.ones(n, dtype=np.int32), np.zeros(n, dtype=np.int32)

    lib = SimpleNamespace(ifci_frozen_core=lambda h, s, X: (None, None, 0.0), CIProblem=lambda *a: a,
                          davidson_opts=lambda precision, **kw: {"precision": precision, **kw},
                          ifci_davidson_expansion=solve)
    torch = SimpleNamespace(cuda=SimpleNamespace(synchronize=lambda dev: None))
    args = SimpleNamespace(max_order=3, compare_fraction=0.05)
    out = bench.paths_sample(lib, torch, None, chain_24_uneven(), None, args, None)
    assert calls == ["fp64e", "fp64", "bf16", "tf32"]
    assert set(out["runs"]) == {"fp64e", "fp64", "bf16_mixed", "tf32_mixed"}
