"""Host-side checks of the down projection shared by pairs of blocks: half of the rows each, the columns both of them produce (no GPU
needed)."""
import numpy as np
import pytest

from sdv_inputs import get_config
from paper_2510_15312_b200.binding import OK, config_from, grid, layout_check, plan


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
    if name == "qwen7b":   # pairs would leave it two ring slots at 16 and 17 rows (below)
        assert down[2] == 1 and down[3] == gu[2] and layout_check(down, gu, blocks) == OK
        return
    pairs = blocks % 2 == 0 and gu[2] % 2 == 0 and 16 * down[0] * gu[2] >= 65536
    assert down[2] == (2 if pairs else 1) and down[2] * down[3] == gu[2]
    assert pairs == (name[0] in "ql" and blocks > 100)
    assert layout_check(down, gu, blocks) == OK


@pytest.mark.parametrize("d,steps,k", [(1024, 28, 3), (1536, 20, 1), (2048, 12, 2), (1536, 8, 7), (896, 4, 8)])
def test_pairs_refuse_no_rows(d, steps, k):
    """A batched step has more rows than a draft of k_max: pairs are taken only where every number of rows fits that single blocks, whose
    operand is half as large, can take.  147 blocks never work in pairs; the largest share has `steps` column steps there and in 148."""
    cc = config_from(get_config("qwen1.5b"), k_max=k)
    cc.d_model, cc.d_ffn = d, 16 * 147 * steps
    for rows in range(1, 33):
        (ops1, single), (ops2, pairs) = plan(cc, 147, rows), plan(cc, 148, rows)
        assert ops1[3][2] == 1 and ops1[2][2] == 147 and ops2[2][2] == 148
        assert pairs[5] >= single[5], (rows, ops2[3])
    assert steps > 4 or ops2[3][2] == 2


@pytest.mark.parametrize("k", [4, 16, 20])
def test_pairs_cost_no_third_ring_slot(k):
    """The 7B shape, whose layers HBM bounds: 16 and 17 rows have three ring slots with single blocks and would have two with pairs.  (147
    blocks never work in pairs; their largest shares are those of 148 to the column step.)"""
    cc = config_from(get_config("qwen7b"), k_max=k)
    for rows in range(1, 33):
        (_, single), (ops, taken) = plan(cc, 147, rows), plan(cc, 148, rows)
        assert ops[3][2] == 1 and min(taken[2], 3) >= min(single[2], 3), rows
        assert taken[2] >= 3 or rows > 17


@pytest.mark.parametrize("sms,clusters,blocks,pairs", [(148, 74, 148, True), (148, 80, 148, True), (148, 73, 148, False), (148, 0, 148, False),
                                                       (147, 73, 146, True), (147, 72, 147, False)])
def test_pairs_only_where_the_device_holds_them(sms, clusters, blocks, pairs):
    """All pairs of a launch have to be on the device at once; single blocks otherwise, on every SM."""
    assert grid(config_from(get_config("qwen1.5b")), sms, clusters) == (blocks, pairs)


@pytest.mark.parametrize("sms", [148, 147, 16, 7, 2, 1])
def test_single_blocks_take_every_sm(sms):
    assert grid(config_from(get_config("tiny")), sms, sms // 2) == (sms, False)
