"""GPU parity of the down projection shared by pairs of blocks, at small depths: shares of one and two column steps side by side, passes of
one and of two accumulators, shares that just make pairs, rows on both sides of an instruction's."""
import numpy as np
import pytest

from oracle import sdv_oracle as O
from sdv_inputs import get_config, make_context, make_weights
from paper_2510_15312_b200.binding import Sdv, config_from, plan
from helpers import COS_TOL, LOGIT_TOL
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


PAIRED = ("tiny", dict(d_model=1024, d_ffn=1088, n_ctx=90, chunk=64))   # 68 shares of a step: 34 pairs


def near(got, want):
    cos = (got * want).sum(1) / (np.linalg.norm(got, axis=1) * np.linalg.norm(want, axis=1))
    assert np.abs(got - want).max() <= LOGIT_TOL and cos.min() >= COS_TOL


def in_pairs(cfg, k_max):
    w, ctx = make_weights(cfg), make_context(cfg)
    s = Sdv(config_from(cfg, k_max=k_max, max_seq=cfg.n_ctx + 80))
    s.load_weights(w)
    assert s.debug_grid()[1]
    return s, w, ctx


@pytest.mark.parametrize("nodes", [3, 15, 16, 20])
def test_tree_verify_in_pairs(nodes):
    cfg = get_config(PAIRED[0]).with_(**PAIRED[1])
    s, w, ctx = in_pairs(cfg, 24)
    ref = O.OracleModel(w)
    T = O.argmax(ref.prefill(ctx, cfg.chunk))
    s.set_parity_mode(True)
    for i in range(0, cfg.n_ctx, cfg.chunk):
        s.prefill_chunk(ctx[i:i + cfg.chunk], is_last=i + cfg.chunk >= cfg.n_ctx)
    s.debug_set_history(list(ctx) + [T], cfg.n_ctx)
    rng = np.random.default_rng(nodes)
    tokens, parent = rng.integers(0, cfg.vocab, nodes).tolist(), [int(rng.integers(0, i + 1)) for i in range(nodes)]
    s.verify_tree(tokens, parent)
    near(s.get_logits(nodes + 1), np.asarray(ref.forward([T] + tokens, cfg.n_ctx, parent=[0] + parent)).reshape(nodes + 1, -1))
    s.close()


@pytest.mark.parametrize("lengths", [(8, 8), (4, 0, 9), (12, 12, 5)])
def test_batched_step_in_pairs(lengths):
    """Sequences of different context and draft lengths in one launch, each against its own oracle: 16, 16 and 32 rows."""
    cfg = get_config(PAIRED[0]).with_(**PAIRED[1])
    lead, w, ctx = in_pairs(cfg, 12)
    seqs = [lead] + [lead.follower() for _ in lengths[1:]]
    rng = np.random.default_rng(sum(lengths))
    want = []
    for i, (s, n) in enumerate(zip(seqs, lengths)):
        own = ctx[:cfg.n_ctx - 17 * i]
        ref = O.OracleModel(w)
        T = O.argmax(ref.prefill(own, cfg.chunk))
        s.set_parity_mode(True)
        for at in range(0, len(own), cfg.chunk):
            s.prefill_chunk(own[at:at + cfg.chunk], is_last=at + cfg.chunk >= len(own))
        s.debug_set_history(list(own) + [T], len(own))
        draft = [int(t) for t in rng.integers(0, cfg.vocab, n)]
        s.debug_set_draft(draft)
        want.append(np.asarray(ref.forward([T] + draft, len(own))).reshape(n + 1, -1))
    Sdv.verify_batch(seqs)
    for s, n, rows in zip(seqs, lengths, want):
        near(s.get_logits(n + 1), rows)
    for s in reversed(seqs):
        s.close()
