"""Host-side checks of the stacked K slices and of the most rows the wide shapes take (no GPU needed)."""
import numpy as np
import pytest

from sdv_inputs import get_config
from paper_2510_15312_b200.binding import OK, config_from, layout_check, plan


@pytest.mark.parametrize("slices", [1, 2, 4, 8])
def test_stacked_slices_cover_each_matrix_once(slices):
    rng = np.random.default_rng(slices)
    for _ in range(60):
        RW = int(rng.integers(1, 8 // slices + 1))
        SK = int(rng.integers(1, 64 // (RW * slices) + 1))
        T, G = int(rng.integers(1, 40)), int(rng.integers(1, 20))
        o = [T, slices * int(rng.integers(1, 20)), min(G, T), 1, RW, SK, 1, slices << 8]
        assert layout_check(o, o, G) == OK, o


@pytest.mark.parametrize("name,k", [("llama3b", 24), ("qwen7b", 20), ("qwen1.5b", 31), ("qwen0.5b", 31)])
def test_most_drafts_of_the_wide_shapes_fit(name, k):
    cfg = get_config(name)
    ops, sp = plan(config_from(cfg, k_max=k), 148, k + 1)
    assert sp[5] == 1 and sp[2] >= 2
    for o in ops:
        assert layout_check(o, ops[2], 148) == OK
