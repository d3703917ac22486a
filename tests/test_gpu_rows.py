"""Which rows of a verify step exist: a draft held on the device may be shorter than the bound the host knows.  What the
read-back calls return, and what the forced commits accept, for the rows past it."""
import numpy as np
import pytest

from sdv_inputs import get_config, make_context, make_weights
from paper_2510_15312_b200.binding import EINVAL, Sdv, SdvError, config_from

pytestmark = pytest.mark.gpu

BOUND = 8              # drafts the host assumes
AGAIN = 1e-2           # the same rows twice: partial sums meet in another order (fp32), a bf16 rounding behind them may flip


@pytest.fixture(scope="module")
def seq():
    cfg = get_config("tiny")
    ctx = make_context(cfg)
    s = Sdv(config_from(cfg, k_max=24))
    s.load_weights(make_weights(cfg))
    for i in range(0, cfg.n_ctx, cfg.chunk):
        s.prefill_chunk(ctx[i:i + cfg.chunk], is_last=i + cfg.chunk >= cfg.n_ctx)
    yield s, cfg, s.kv_len()
    s.close()


def short_draft(s, tokens):
    """A draft of these tokens on the device; the host only knows that it has at most BOUND."""
    s.debug_set_draft(tokens)
    s.extend_draft(BOUND, fetch=False)


def rows_of(s, cfg, L):
    return (s.get_logits(BOUND + 1), s.debug_read_hidden(BOUND + 1),
            *[s.debug_read_kv(cfg.n_layers - 1, which, L, BOUND + 1) for which in (0, 1)])


@pytest.mark.parametrize("n", [0, 3, BOUND])
def test_parity_mode_stores_every_row_up_to_the_bound(seq, n):
    """Rows past the draft are those of padding tokens 0, not what an earlier step left."""
    s, cfg, L = seq
    s.rollback(L)
    s.set_parity_mode(True)
    draft = [int(t) for t in np.random.default_rng(n).integers(1, cfg.vocab, n)]
    s.verify(draft + [0] * (BOUND - n))
    want = rows_of(s, cfg, L)
    s.verify([7] * 24)                       # something else in every buffer
    short_draft(s, draft)
    y, a = s.verify(None)
    for got, ref in zip(rows_of(s, cfg, L), want):
        assert np.abs(got - ref).max() <= AGAIN * max(1.0, np.abs(ref).max())
    s.set_parity_mode(False)                 # and without it the draft's own rows are the same
    s.rollback(L)
    short_draft(s, draft)
    y2, a2 = s.verify(None)
    assert list(y2[:n + 1]) == list(y[:n + 1]) and a2 == a
    assert np.abs(s.debug_read_hidden(n + 1) - want[1][:n + 1]).max() <= AGAIN * max(1.0, np.abs(want[1]).max())


@pytest.mark.parametrize("parity", [False, True])
def test_forced_commits_stop_at_the_draft(seq, parity):
    """No rows beyond the verified draft can be committed, whatever bound the host had for it."""
    s, cfg, L = seq
    s.rollback(L)
    s.set_parity_mode(parity)
    short_draft(s, [5, 6, 7])
    s.verify(None, fetch=False)
    for a in (4, BOUND, BOUND + 1):
        with pytest.raises(SdvError) as e:
            s.debug_force_commit(a, 9)
        assert e.value.code == EINVAL
    assert s.kv_len() == L
    s.debug_force_commit(3, 9)
    assert s.kv_len() == L + 4
    s.rollback(L)
    s.draft_tree(0, BOUND, fetch=False)      # no calibration: a tree of no nodes
    s.verify_tree(fetch=False)
    for path in ([1], [BOUND]):
        with pytest.raises(SdvError) as e:
            s.debug_force_commit_tree(path, 9)
        assert e.value.code == EINVAL
    s.debug_force_commit_tree([], 9)
    assert s.kv_len() == L + 1
    s.set_parity_mode(False)


def test_verified_tokens_are_those_of_the_rows_that_exist(seq):
    """sdv_get_verified writes draft length + 1 tokens, as sdv_verify does (the binding hands in zeros)."""
    s, cfg, L = seq
    s.rollback(L)
    s.verify([7] * 24)
    short_draft(s, [5, 6])
    y, a = s.verify(None)
    got, a2 = s.get_verified()
    assert a2 == a and list(got[:3]) == list(y[:3]) and not got[3:].any()


def test_a_device_verify_behind_a_host_verify_looks_at_its_own_rows(seq):
    """Without a draft of the device's own a step runs the pending token's row alone, whatever draft the verify before was
    given; where there was one, the draft handed in has taken its place."""
    s, cfg, L = seq
    s.rollback(L)
    y, _ = s.verify([])
    story = [int(y[0])]
    for _ in range(5):                       # the model's own continuation: accepted whole
        y, a = s.verify(story)
        assert a == len(story)
        story.append(int(y[len(story)]))
    s.rollback(L)
    assert s.verify(story)[1] == len(story)
    y, a = s.verify(None)
    assert a == 0 and int(y[0]) == story[0]
    assert s.commit()[0] == story[:1]
    s.rollback(L)
    s.debug_set_draft(story[:2])
    s.verify(story)
    y, a = s.verify(None)
    assert a == len(story) and [int(t) for t in y[:a]] == story
    assert s.commit()[0][:a] == story
    for again in (lambda: s.step(None, 0)[0], lambda: Sdv.verify_batch([s]) == [0] and s.commit()[0]):
        s.rollback(L)
        s.verify(story)
        assert again() == story[:1]
