"""Host-side checks of the down projection shared by pairs of blocks: half of the rows each, the columns both of them produce (no GPU
needed)."""
import numpy as np
import pytest

from sdv_inputs import get_config
from paper_2510_15312_b200.binding import OK, config_from, layout_check, plan


def test_pairs_cover_each_matrix_once():
    rng = np.random.default_rng(2)
    for _ in range(150):
        G = 2 * int(rng.integers(1, 11))
        units = int(rng.integers(2, 60))
        shares = min(G, units) // 2 * 2
        gu = [2 * units, int(rng.integers(1, 20)), shares, 1, 16, 4, 2, 0]
        down = [int(rng.integers(2, 40)), units, 2, shares // 2, 16, int(rng.integers(1, 5)), 1, 1]
        assert layout_check(gu, gu, G) == OK
        assert layout_check(down, gu, G) == OK, (down, gu, G)


@pytest.mark.parametrize("name,k", [("tiny", 31), ("mini_gqa", 31), ("qwen0.5b", 31), ("qwen1.5b", 31), ("llama3b", 24), ("qwen7b", 20)])
@pytest.mark.parametrize("blocks", [148, 132, 7])
def test_who_takes_pairs(name, k, blocks):
    """Pairs where the shares are even in number and their partial sums many; single blocks otherwise; either covers the matrix."""
    ops, sp = plan(config_from(get_config(name), k_max=k), blocks, 1)
    gu, down = ops[2], ops[3]
    pairs = blocks % 2 == 0 and gu[2] % 2 == 0 and 16 * down[0] * gu[2] >= 65536
    assert down[2] == (2 if pairs else 1) and down[2] * down[3] == gu[2]
    assert pairs == (name[0] in "ql" and blocks > 100)
    assert layout_check(down, gu, blocks) == OK
