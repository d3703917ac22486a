"""GPU parity at the sizes where tiles, chunks and shares have their edges: prefill sub-chunks around the tile sizes, key
ranges of several chunks, wide rows, operands of many rows, and the stand-alone GEMM's row groups and clusters."""
import numpy as np
import pytest

from oracle import sdv_oracle as O
from sdv_inputs import bf16_bits_to_f32, f32_to_bf16_bits, get_config, make_context, make_weights
from paper_2510_15312_b200.binding import OK, Sdv, config_from, gemm_noalloc, plan
from helpers import COS_TOL, LOGIT_TOL

pytestmark = pytest.mark.gpu


def check(cfg, drafts, calib=0):
    """Prefill in cfg.chunk tokens, then one verify step per draft length over the same cache, against the oracle."""
    w, ctx = make_weights(cfg), make_context(cfg)
    ref = O.OracleModel(w)
    last = ref.prefill(ctx, cfg.chunk)
    s = Sdv(config_from(cfg))
    try:
        s.load_weights(w)
        s.set_parity_mode(True)
        if calib:
            s.set_calibration(calib)
        for i in range(0, cfg.n_ctx, cfg.chunk):
            s.prefill_chunk(ctx[i:i + cfg.chunk], is_last=i + cfg.chunk >= cfg.n_ctx)
        for which, name in ((0, "k"), (1, "v")):
            kv, want = s.debug_read_kv(cfg.n_layers - 1, which, 0, cfg.n_ctx), ref.kv_view(name)[cfg.n_layers - 1][:, :cfg.n_ctx]
            assert np.abs(kv - want).max() <= 0.02 * np.abs(want).max() + 1e-3, name
        if calib:
            rows = O.OracleModel(w).prefill_all_logits(ctx, cfg.chunk)
            succ, _ = s.get_calibration(cfg.n_ctx)
            for p in range(cfg.n_ctx):
                floor = np.sort(rows[p])[-calib] - 2 * LOGIT_TOL
                assert len(set(succ[p].tolist())) == calib and all(rows[p][t] >= floor for t in succ[p]), p
        T = O.argmax(last)
        rng = np.random.default_rng(cfg.n_ctx)
        for n in drafts:
            draft = [int(t) for t in rng.integers(0, cfg.vocab, n)]
            s.debug_set_history(list(ctx) + [T], cfg.n_ctx)
            s.verify(draft)
            got = s.get_logits(n + 1)
            want = np.asarray(ref.forward([T] + draft, cfg.n_ctx)).reshape(n + 1, -1)
            assert np.abs(got - want).max() <= LOGIT_TOL, n
            cos = (got * want).sum(1) / (np.linalg.norm(got, axis=1) * np.linalg.norm(want, axis=1))
            assert cos.min() >= COS_TOL, n
    finally:
        s.close()


# around 16 rows (the small-row kernel below), 128 (rows per SM, keys per block), 256 (rows per pair), beyond 1024 (two
# sub-chunks); every remainder chunk differs from the full one.  The vocabulary is no multiple of a tile.
@pytest.mark.parametrize("name,n_ctx,chunk", [("mini_hd128", 46, 15), ("mini_hd128", 33, 16), ("tiny", 35, 17), ("mini_gqa", 300, 127),
                                              ("mini_hd128", 300, 128), ("tiny", 387, 129), ("mini_gqa", 520, 255),
                                              ("mini_hd128", 513, 256), ("mini_gqa", 700, 257), ("mini_hd128", 1025, 1025),
                                              ("mini_gqa", 1100, 1040)])
def test_prefill_and_calibration_at_tile_edges(name, n_ctx, chunk):
    check(get_config(name).with_(n_ctx=n_ctx, chunk=chunk), (0, 4), calib=3)


# key chunks of 128 and their edges; ranges of several chunks (many KV heads leave few blocks to each); row counts on
# both sides of every operand and accumulator step; K slices of the q|k|v share; rows of several segments and
# beyond ten of them; many partial results per row
@pytest.mark.parametrize("name,over,drafts", [
    ("mini_gqa", dict(n_ctx=127, k=31), (0, 1, 7, 8, 31)),
    ("mini_hd128", dict(n_ctx=128, k=31), (0, 15, 16, 23, 24, 31)),
    ("tiny", dict(n_ctx=129, k=31), (0, 16, 20, 31)),
    ("tiny", dict(n_q_heads=32, n_kv_heads=32, n_ctx=1100, k=8), (0, 3, 8)),
    ("mini_hd128", dict(n_q_heads=24, n_kv_heads=24, n_ctx=1700, k=8), (0, 8)),
    ("mini_hd128", dict(n_q_heads=8, n_kv_heads=1, n_ctx=2500, k=24), (0, 8, 23, 24)),
    ("tiny", dict(d_model=2112, d_ffn=2112, n_ctx=70, k=16), (0, 8, 16)),
    ("mini_gqa", dict(d_model=4160, n_ctx=40, k=8), (0, 8)),
    ("tiny", dict(n_layers=1, d_model=10304, n_q_heads=2, n_kv_heads=1, d_ffn=128, vocab=528, n_ctx=24, k=4), (0, 4)),
])
def test_verify_at_chunk_and_share_edges(name, over, drafts):
    check(get_config(name).with_(**over), drafts)


def test_passes_of_nine_and_eight_tiles():
    """Shares of 17 row tiles are walked in passes of nine and eight: two accumulators and one side by side.  Here the LM head's (half of the blocks;
    the others have 16 tiles in one pass)."""
    cfg = get_config("tiny").with_(vocab=16 * (148 * 16 + 74), n_ctx=40, k=16)
    lm = plan(config_from(cfg), 148, 1)[0][4]
    assert lm[0] == 148 * 16 + 74 and lm[2] == 148 and lm[4] == 16
    check(cfg, (0, 8, 16))


@pytest.mark.parametrize("M", [1, 8, 9, 16, 17, 24, 25, 32])
def test_gemm_row_groups_and_clusters(M):
    """Tiles of 8 token rows; one 32-column step per warp and several; few and many row tiles (clusters of 8 down to 1)."""
    import torch
    for N, K in ((16, 64), (16, 4096), (272, 1088), (2416, 384), (4080, 64)):
        rng = np.random.default_rng(M * 7919 + N + K)
        x, wb = rng.standard_normal((M, K)).astype(np.float32), f32_to_bf16_bits(rng.standard_normal((N, K)).astype(np.float32))
        y = torch.full((M, N), float("nan"), device="cuda")
        assert gemm_noalloc(torch.from_numpy(x).cuda(), torch.from_numpy(wb.view(np.int16)).cuda(), y) == OK
        np.testing.assert_allclose(y.cpu().numpy(), O.matmul(bf16_bits_to_f32(f32_to_bf16_bits(x)), wb), rtol=0, atol=2e-5 * np.sqrt(K))
