"""The autotuner's own grid times two wave budgets only where they can differ
(no GPU)."""
import pytest

from paper_2307_10675_gb300 import autotune


@pytest.mark.parametrize("precision,budgets", [("fp64", 1), ("fp64e", 1), ("bf16", 2), ("tf32", 2), ("fp32", 2)])
def test_budgets_timed(precision, budgets):
    grid = autotune.default_grid(precision)
    assert len(grid["det_budget"]) == budgets and grid["det_budget"][0] == 1 << 31
    assert grid["max_space"] == autotune.DEFAULT_GRID["max_space"]
    assert len(autotune.DEFAULT_GRID["det_budget"]) == 2   # the table itself stays whole
