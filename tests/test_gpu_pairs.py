"""GPU parity of the down projection shared by pairs of blocks, at small depths: shares of one and two column steps side by side, passes of
one and of two accumulators, shares that just make pairs, rows on both sides of an instruction's."""
import pytest

from sdv_inputs import get_config
from paper_2510_15312_b200.binding import Sdv, config_from, plan
from test_gpu_shapes import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,over,drafts", [
    ("tiny", dict(d_model=1024, d_ffn=1024, n_ctx=40, k=31), (0, 8, 16, 31)),      # 64 shares of a step: 64 K sums; 32 tiles: two passes of 16
    ("tiny", dict(d_model=1088, d_ffn=2432, n_ctx=70, k=31), (0, 15, 31)),         # 148 shares, four of them of two steps; 34 tiles in three passes
    ("mini_hd128", dict(d_model=448, d_ffn=7168, n_ctx=50, k=16), (0, 7, 16)),     # 148 shares of three and four steps; 14 tiles: one pass
    ("mini_gqa", dict(d_model=704, d_ffn=1536, n_ctx=33, k=8), (0, 8)),            # 96 shares; 22 tiles in two passes
])
def test_verify_and_prefill_tiles_in_pairs(name, over, drafts):
    cfg = get_config(name).with_(chunk=13, **over)     # chunks of 13 rows take the verify kernel without its LM head
    assert plan(config_from(cfg), 148, 1)[0][3][2] == 2
    check(cfg, drafts)


def test_a_context_takes_the_pairs_its_plan_has():
    """The device is asked how many pairs it holds: all of them here, so that no context falls back to single blocks unseen."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for name, over, pairs in (("tiny", dict(d_model=1024, d_ffn=1024), True), ("mini_hd128", dict(d_model=448, d_ffn=7168), True), ("tiny", dict(), False)):
        s = Sdv(config_from(get_config(name).with_(**over)))
        assert s.debug_grid() == (sms, pairs)
        s.close()
