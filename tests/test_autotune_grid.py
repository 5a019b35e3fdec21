"""The autotuner's own grid times two wave budgets only where they can differ,
and a candidate within its margin of the best does not replace it (no GPU)."""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2307_10675_gb300 import autotune


@pytest.mark.parametrize("precision,budgets", [("fp64", 1), ("fp64e", 1), ("bf16", 2), ("tf32", 2), ("fp32", 2)])
def test_budgets_timed(precision, budgets):
    grid = autotune.default_grid(precision)
    assert len(grid["det_budget"]) == budgets and grid["det_budget"][0] == 1 << 31
    assert grid["max_space"] == autotune.DEFAULT_GRID["max_space"]
    assert len(autotune.DEFAULT_GRID["det_budget"]) == 2   # the table itself stays whole


@pytest.mark.parametrize("seconds,chosen", [({12: 2.986, 10: 2.985, 16: 3.4}, 12), ({12: 2.986, 10: 2.80, 16: 2.79}, 10),
                                            ({12: 3.0, 10: 3.1, 16: 2.5}, 16)])
def test_a_tie_keeps_the_incumbent(monkeypatch, seconds, chosen):
    monkeypatch.setattr(autotune, "_problems", lambda handle, system, sets: [])
    monkeypatch.setattr(autotune, "_time", lambda handle, probs, opts, warm: (seconds[opts.max_space], np.zeros(1)))
    monkeypatch.setattr(autotune.torch.cuda, "get_device_name", lambda device: "none")
    system = SimpleNamespace(body_offset=[0, 2, 4], nbody=2)
    out = autotune.autotune(SimpleNamespace(device=0), system, [(0, 1)], grid={"max_space": [12, 10, 16]})
    assert out["params"] == {"max_space": chosen}
    assert len(out["table"]) == 3
