"""bench.py reports what runs (no GPU): the solver of the path comparison (the
library is a stand-in that records the calls) and the operations of a sigma."""
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


def test_sigma_flops_of_the_fp64_path():
    # H of CAS(6e,13o), row by row of one determinant's excitations: the diagonal, 30 singles and
    # 135 doubles of each spin; 33 excitations (diagonal ones among them) of each spin at once
    assert bench.sigma_flops("fp64", 13, 3, 91) == 2.0 * 286 ** 2 * (33 ** 2 + 2 * 166)
    assert bench.sigma_flops("bf16", 13, 3, 91) == 2.0 * 286 ** 2 * 91 ** 2
    assert bench.sigma_flops("fp64e", 13, 3, 91) == 2.0 * 286 ** 2 * 91 * 33
