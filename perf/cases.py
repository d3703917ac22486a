"""The work a user of this library has it do, as timed cases: requests through the public entry points at the
model shapes of sdv_inputs/configs.py, with synthetic weights whose greedy predictions are as clear-cut as a
trained model's and contexts that repeat what the model goes on to say, so that drafts are accepted in part.

Kinds of case
  gemm       the stand-alone GEMM on device tensors (sdv_gemm_noalloc), as a plug-in calls it
  step       decoding with the host in the loop: draft, then sdv_step per step (drafts in, tokens out)
  decode     decoding in runs of steps without the host in between (sdv_decode_steps)
  tree       one step with a calibrated tree draft: sdv_draft_tree, sdv_verify_tree, sdv_commit
  batch      one verify step shared by several sequences: sdv_draft each, sdv_verify_batch, sdv_commit each
  prefill    a new request on loaded weights: its context in chunks, then the first verify step
  calibrate  the same with in-context calibration, whose tables come back to the host
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2510_15312_b200 import binding
from paper_2510_15312_b200.binding import Sdv, config_from
from sdv_inputs import get_config

# Draft lengths a shape can be given: the k_max + 1 token rows have to fit in shared memory beside the weight ring.
MOST_DRAFTS = {"tiny": 31, "qwen0.5b": 31, "qwen1.5b": 31, "llama3b": 24, "qwen7b": 20}
EXTENSION_LIFE = 4   # verify steps a segment of rejected drafts is kept for
TOP_B = 2            # successors sampled per context position by the calibration
# A token's two likely successors: shares of the prediction's strength (their squares sum to 1).
SUCCESSOR_STRENGTH = (0.84, 0.54)


def listed():
    return [
        # one projection of a small adapter, called from a plug-in that may not allocate: launches and host work count
        dict(name="gemm 9 x 640 x 768", kind="gemm", rows=9, n=640, k=768),
        # the smallest model, host in the loop: latency of one step
        dict(name="step tiny k4", kind="step", model="tiny", ctx=512, k=4, steps=4, bias=False),
        # the usual decoding loop at the small, the middle and the large shapes; drafts as the configurations name them
        dict(name="decode 0.5b k8", kind="decode", model="qwen0.5b", ctx=1024, k=8, steps=8, extend=0, bias=False),
        dict(name="decode 1.5b k8", kind="decode", model="qwen1.5b", ctx=2048, k=8, steps=8, extend=0, bias=False),
        dict(name="decode 3b k16", kind="decode", model="llama3b", ctx=4096, k=16, steps=4, extend=0, bias=False),
        dict(name="decode 7b k4", kind="decode", model="qwen7b", ctx=8192, k=4, steps=4, extend=0, bias=False),
        # rejected drafts kept and appended to later ones: the widest verify step, over a short context of odd length
        dict(name="decode 1.5b extended to 31", kind="decode", model="qwen1.5b", ctx=777, k=8, steps=8, extend=31, bias=True),
        # calibrated tree drafts
        dict(name="tree 1.5b 20 nodes", kind="tree", model="qwen1.5b", ctx=1500, k=8, nodes=20, bias=False),
        # three requests served together
        dict(name="batch 1.5b 3 x k8", kind="batch", model="qwen1.5b", ctx=2048, k=8, sequences=3, bias=False),
        # new requests: the configurations' chunk length at the middle and the large shape
        dict(name="prefill 1.5b 2048", kind="prefill", model="qwen1.5b", ctx=2048, chunk=256, k=8, bias=False),
        dict(name="prefill 7b 2048", kind="prefill", model="qwen7b", ctx=2048, chunk=256, k=4, bias=True),
        # a short request with calibration, ragged chunks
        dict(name="calibrate 0.5b 700", kind="calibrate", model="qwen0.5b", ctx=700, chunk=150, k=8, bias=True),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gemm", "step", "decode", "decode", "decode", "tree", "batch", "prefill", "prefill", "calibrate"])
    if kind == "gemm":
        k = 64 * _log(rng, 2, 64)
        return dict(kind=kind, rows=_log(rng, 1, 32), n=16 * _log(rng, 4, min(256, (1 << 20) // k // 16)), k=k)
    bias = rng.random() < 0.5
    if kind == "step":
        model = rng.choice(["tiny", "qwen0.5b", "qwen1.5b"])
        return dict(kind=kind, model=model, ctx=_log(rng, 64, 4096), k=_log(rng, 1, 16), steps=rng.randint(2, 6), bias=bias)
    if kind == "decode":
        model = rng.choice(["qwen0.5b", "qwen1.5b", "llama3b", "qwen7b"])
        k = _log(rng, 1, 16)
        extend = rng.randint(k, MOST_DRAFTS[model]) if rng.random() < 0.25 else 0
        return dict(kind=kind, model=model, ctx=_log(rng, 100, 8192), k=k, steps=rng.randint(2, 8), extend=extend, bias=bias)
    if kind == "tree":
        return dict(kind=kind, model=rng.choice(["qwen0.5b", "qwen1.5b"]), ctx=_log(rng, 200, 2048), k=rng.randint(0, 12),
                    nodes=rng.randint(4, 31), bias=bias)
    if kind == "batch":
        n = rng.randint(2, 6)
        return dict(kind=kind, model=rng.choice(["qwen0.5b", "qwen1.5b", "llama3b"]), ctx=_log(rng, 200, 4096), k=_log(rng, 1, 24 // n - 1),
                    sequences=n, bias=bias)
    if kind == "calibrate":
        return dict(kind=kind, model=rng.choice(["qwen0.5b", "qwen1.5b"]), ctx=_log(rng, 100, 1500), chunk=_log(rng, 48, 512), k=8, bias=bias)
    model = rng.choice(["qwen0.5b", "qwen1.5b", "llama3b", "qwen7b"])
    return dict(kind=kind, model=model, ctx=_log(rng, 60, {"qwen7b": 2048, "llama3b": 4096}.get(model, 6000)), chunk=_log(rng, 32, 1024),
                k=rng.randint(1, 8), bias=bias)


# ------------------------------------------------------------------------------------------ inputs
def _weights(cfg, seed):
    """Random decoder weights on the GPU, scaled as sdv_inputs scales its own.  The LM head is built from the
    embedding so that every token has two likely successors (the permutations `nexts`), strongest first."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    d, f, hd = cfg.d_model, cfg.d_ffn, cfg.head_dim
    nq, nkv = cfg.n_q_heads * hd, cfg.n_kv_heads * hd
    s = 1.0 / math.sqrt(d)

    def matrix(rows, cols, std):
        return torch.empty((rows, cols), dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=gen)

    def vector(n, mean, std):
        return torch.empty(n, dtype=torch.float32, device="cuda").normal_(mean, std, generator=gen)

    emb = matrix(cfg.vocab, d, s)
    nexts = [torch.randperm(cfg.vocab, generator=gen, device="cuda") for _ in SUCCESSOR_STRENGTH]
    head = torch.zeros((cfg.vocab, d), dtype=torch.float32, device="cuda")
    for nx, a in zip(nexts, SUCCESSOR_STRENGTH):
        head[nx] += a * emb.float()
    layers = []
    for _ in range(cfg.n_layers):
        layers.append(SimpleNamespace(
            wq=matrix(nq, d, math.sqrt(cfg.qk_var) * s), wk=matrix(nkv, d, math.sqrt(cfg.qk_var) * s), wv=matrix(nkv, d, s),
            wo=matrix(d, nq, cfg.resid_scale * s / math.sqrt(nq)), wg=matrix(f, d, s), wu=matrix(f, d, s),
            wd=matrix(d, f, cfg.resid_scale * s / math.sqrt(f)), norm1=vector(d, 1.0, 0.1), norm2=vector(d, 1.0, 0.1),
            bq=vector(nq, 0.0, 0.02) if cfg.qkv_bias else None, bk=vector(nkv, 0.0, 0.02) if cfg.qkv_bias else None,
            bv=vector(nkv, 0.0, 0.02) if cfg.qkv_bias else None))
    return SimpleNamespace(emb=emb, lm_head=head.to(torch.bfloat16), final_norm=vector(d, 1.0, 0.1), layers=layers), nexts[0].cpu().numpy()


def _context(vocab, n, nxt, rng):
    """A request of n tokens: passages of a story the model itself would tell (each token followed by its likeliest
    successor) between stretches of other tokens (Zipf over the vocabulary); it ends inside the story."""
    story = [int(rng.integers(vocab))]
    while len(story) < 400:
        story.append(int(nxt[story[-1]]))
    ids = np.minimum(rng.zipf(1.3, size=n) - 1, vocab - 1) * 7919 % vocab
    out = []
    while len(out) < n:
        m = int(rng.integers(4, 25))
        if rng.random() < 0.6:
            at = int(rng.integers(0, 380))
            out += story[at:at + m]
        else:
            out += [int(t) for t in ids[len(out):len(out) + m]]
    at = int(rng.integers(8, 100))
    tail = story[max(0, at - 8):at][-n:]
    return np.array(out[:n - len(tail)] + tail, dtype=np.int32), [int(t) for t in story[at:]]


def _model(case, extra_rows, k_max):
    cfg = get_config(case["model"]).with_(tied_lm_head=False, qkv_bias=bool(case["bias"]))
    return cfg, config_from(cfg, k_max=k_max, max_seq=case["ctx"] + extra_rows + 2 * k_max + 16)


def _prefill(seq, tokens, chunk):
    for i in range(0, len(tokens), chunk):
        seq.prefill_chunk(tokens[i:i + chunk], is_last=i + chunk >= len(tokens))


def prepare(case, seed):
    """Inputs in hand: device tensors for the stand-alone GEMM, otherwise a context with loaded weights and, where
    the case starts behind the prefill, the request's KV cache."""
    rng = np.random.default_rng([seed, 17])
    if case["kind"] == "gemm":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn((case["rows"], case["k"]), generator=gen, device="cuda")
        w = torch.randn((case["n"], case["k"]), generator=gen, device="cuda").mul_(1 / math.sqrt(case["k"])).to(torch.bfloat16)
        return SimpleNamespace(case=case, x=x, w=w, y=torch.empty((case["rows"], case["n"]), device="cuda"))
    kind, ctx = case["kind"], case["ctx"]
    rows = max(case["k"], case.get("extend", 0), case.get("nodes", 0))
    cfg, ccfg = _model(case, (case.get("steps", 1) + 1) * (rows + 1), rows)
    weights, nxt = _weights(cfg, seed)
    lead = Sdv(ccfg)
    lead.load_weights(weights)
    del weights
    st = SimpleNamespace(case=case, seq=lead)
    if kind in ("prefill", "calibrate"):
        st.tokens, follow = _context(cfg.vocab, ctx, nxt, rng)
        st.draft = follow[1:1 + case["k"]]
        return st
    st.seqs = [lead] + [lead.follower() for _ in range(case.get("sequences", 1) - 1)]
    if kind == "tree":
        lead.set_calibration(TOP_B)
    st.lengths = []
    for i, q in enumerate(st.seqs):
        tokens, _ = _context(cfg.vocab, max(32, ctx - i * (ctx // 8)), nxt, rng)
        _prefill(q, tokens, cfg.chunk)
        st.lengths.append(len(tokens))
    return st


# ------------------------------------------------------------------------------------------ one pass
def _ints(v, room=0):
    """Whole numbers as an array; where their count depends on what was accepted, filled up to `room` entries with -1."""
    out = np.full(max(room, len(v)), -1, dtype=np.int32)
    out[:len(v)] = v
    return out


def run(st):
    """One pass.  Where a case decodes, the sequence is first rolled back to its request, so that every pass does the
    same work; tokens, lengths and the final hidden state of the rows that count come back."""
    c, kind = st.case, st.case["kind"]
    if kind == "gemm":
        rc = binding.gemm_noalloc(st.x, st.w, st.y)
        if rc != binding.OK:
            raise RuntimeError("gemm_noalloc: %d" % rc)
        return st.y
    if kind == "prefill":
        q = st.seq.follower()
        _prefill(q, st.tokens, c["chunk"])
        y, a = q.verify(st.draft)
        out = dict(y=_ints(y[:len(st.draft) + 1]), accepted=a, kv_len=q.kv_len(), hidden=q.debug_read_hidden(len(st.draft) + 1))
        q.close()
        return out
    if kind == "calibrate":
        q = st.seq.follower()
        q.set_calibration(TOP_B)
        _prefill(q, st.tokens, c["chunk"])
        succ, occ = q.get_calibration(len(st.tokens))
        y, a = q.verify(st.draft)
        out = dict(succ=succ, occ=occ, y=_ints(y[:len(st.draft) + 1]), accepted=a, hidden=q.debug_read_hidden(len(st.draft) + 1))
        q.close()
        return out
    for q, n in zip(st.seqs, st.lengths):
        q.rollback(n)
    q = st.seq
    if kind == "step":
        tokens, draft, kv = [], q.draft(c["k"]), 0
        for _ in range(c["steps"]):
            emitted, draft, kv = q.step(draft, c["k"])
            tokens += emitted
        return dict(tokens=_ints(tokens, c["steps"] * (c["k"] + 1)), next_draft=_ints(draft, c["k"]), kv_len=kv, hidden=q.debug_read_hidden(1))
    if kind == "decode":
        tokens, kv = q.decode_steps(c["k"], c["steps"], ext_max_total=c["extend"], ext_max_life=EXTENSION_LIFE)
        return dict(tokens=_ints(tokens, c["steps"] * (max(c["k"], c["extend"]) + 1)), kv_len=kv, hidden=q.debug_read_hidden(1))
    if kind == "tree":
        nodes, parent = q.draft_tree(c["k"], c["nodes"])
        y, path = q.verify_tree()
        hidden = np.zeros((c["nodes"] + 1, q.cfg.d_model), dtype=np.float32)
        hidden[:len(nodes) + 1] = q.debug_read_hidden(len(nodes) + 1)
        emitted, kv = q.commit()
        room = c["nodes"] + 1
        return dict(nodes=_ints(nodes, room), parent=_ints(parent, room), y=_ints(y[:len(nodes) + 1], room), path=_ints(path, room),
                    emitted=_ints(emitted, room), kv_len=kv, hidden=hidden)
    for s in st.seqs:
        s.draft(c["k"], fetch=False)
    accepted = Sdv.verify_batch(st.seqs)
    hidden = q.debug_read_hidden(1)
    done = [s.commit() for s in st.seqs]
    return dict(accepted=_ints(accepted), emitted=_ints([t for e, _ in done for t in e], len(done) * (c["k"] + 1)), kv_len=_ints([kv for _, kv in done]), hidden=hidden)


# ------------------------------------------------------------------------------------------ what a pass cannot do without
def _step_work(cfg, rows, length):
    """One forward pass over `rows` rows at KV length `length`: every linear weight and the cache read once."""
    return (2.0 * cfg.linear_params() + cfg.kv_bytes_per_token() * (length + rows),
            rows * (2.0 * cfg.linear_params() + 4.0 * cfg.n_layers * cfg.n_q_heads * cfg.head_dim * length))


def work(case):
    if case["kind"] == "gemm":
        m, n, k = case["rows"], case["n"], case["k"]
        return dict(bytes=4.0 * m * k + 2.0 * n * k + 4.0 * m * n, flops=2.0 * m * n * k)
    cfg, n = get_config(case["model"]), case["ctx"]
    if case["kind"] in ("step", "decode"):
        b, f = _step_work(cfg, max(case["k"], case.get("extend", 0)) + 1, n)
        return dict(bytes=b * case["steps"], flops=f * case["steps"])
    if case["kind"] == "tree":
        b, f = _step_work(cfg, case["nodes"] + 1, n)
        return dict(bytes=b, flops=f)
    if case["kind"] == "batch":
        m = case["sequences"]
        b, f = _step_work(cfg, m * (case["k"] + 1), n)
        return dict(bytes=b + (m - 1) * cfg.kv_bytes_per_token() * n, flops=f)
    # a request: each chunk is a call of its own and reads the layers' weights and the cache so far
    head = cfg.vocab * cfg.d_model
    b, f = _step_work(cfg, case["k"] + 1, n)
    for at in range(0, n, case["chunk"]):
        b += 2.0 * (cfg.linear_params() - head) + cfg.kv_bytes_per_token() * min(n, at + case["chunk"])
    f += 2.0 * n * (cfg.linear_params() - head) + 2.0 * cfg.n_layers * cfg.n_q_heads * cfg.head_dim * float(n) * n
    if case["kind"] == "calibrate":
        b += 2.0 * head * -(-n // case["chunk"])
        f += 2.0 * n * head
    return dict(bytes=b, flops=f)


def tolerance(case):
    """Tokens, lengths and drafts are exact: the predictions are far apart.  Hidden states pass through bf16 operands
    and a bf16 KV cache in every layer; the second successor of a few positions is a near tie."""
    if case["kind"] == "gemm":
        return {"rel": 1e-5}
    if case["kind"] == "calibrate":
        return {"rel": 1e-2, "differ": 1e-2}
    return {"rel": 1e-2}
