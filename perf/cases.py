"""The work that users of the library have it do, as cases that can be timed and compared.

Every case goes through the public binding (`paper_2404_08698_b200.binding`, one function per C entry point).  Decoders come
in the repository's shapes: tiny (2 layers x 256), 1.1B (22 x 2048, 8 query heads per kv head, head dimension 64), 7B
(32 x 4096, head dimension 128) and 13B (5120 wide).  `depth` cuts the number of layers: where a batch of eight 13B sequences is
measured, a quarter of the depth does per layer exactly what the whole model does.

The weights are dense and random, but the model's greedy continuation is known and far from every tie: token t < S embeds near the
unit vector e_t, the LM head holds near-unit rows that read dimension t for the token pi(t), pi one cycle through 0..S-1, and the
layers add a spread of a few percent per dimension to the residual stream.  So attention, FFN and cache all shape the logits, while
the tokens - and with them the drafts, the acceptance and the number of steps - are the same for every correct implementation.
Prompts walk the cycle with each token replaced at random with probability `corrupt`, which sets how often an n-gram draft is right
(0.39: about one draft in five, as in summaries; 0.15: about three in five, as in code).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2404_08698_b200 import binding as A

#           layers, d_model, query heads, kv heads, head dim, d_ffn, vocab, tokens on the cycle
SHAPES = {
    "tiny": (2, 256, 4, 4, 64, 688, 4096, 256),
    "1b": (22, 2048, 32, 4, 64, 5632, 32000, 2048),
    "7b": (32, 4096, 32, 32, 128, 11008, 32000, 4096),
    "13b": (40, 5120, 40, 40, 128, 13824, 32000, 4096),
}


def shape_of(case: dict) -> SimpleNamespace:
    L, d, hq, hkv, hd, f, v, s = SHAPES[case["model"]]
    return SimpleNamespace(n_layers=case.get("depth", L), d_model=d, n_q_heads=hq, n_kv_heads=hkv, head_dim=hd, d_ffn=f, vocab=v,
                           rope_theta=1.0e4, rms_eps=1.0e-5, S=s)


# ---- the cases ------------------------------------------------------------------------------------------------------------
def listed() -> list[dict]:
    return [
        # A program with its own model keeps the n-gram module beside it: Initialize with a prompt, then after every step of that
        # model an update with the one to six tokens it confirmed and a draft.  The smallest calls there are: latency only.
        dict(name="ngram_calls", kind="ngram", prompt=512, rounds=24, K=5, n_max=5, policy=0, corrupt=0.25),
        # The whole loop on a tiny model (fp32 weights handed over): launches and hand-overs between kernels, no bandwidth.
        dict(name="tiny_generate", kind="generate", model="tiny", prompt=128, new=64, K=4, n_max=3, policy=0, corrupt=0.2),
        # Generation on a 1.1B model with code-like acceptance, one graph launch for the whole loop.
        dict(name="1b_generate", kind="generate", model="1b", prompt=512, new=96, K=5, n_max=5, policy=0, corrupt=0.25),
        # The flagship: a summarisation-shaped request on a 7B model.
        dict(name="7b_generate", kind="generate", model="7b", prompt=1536, new=128, K=5, n_max=5, policy=0, corrupt=0.39),
        # A short question with an odd length, plain greedy decoding (K = 0): the short prompt pass and the 1-row step.
        dict(name="7b_short_greedy", kind="generate", model="7b", prompt=77, new=24, K=0, n_max=5, policy=0, corrupt=0.39),
        # The loop driven from a host program (own stop rules between steps): draft, verify, update, one call each.
        dict(name="1b_host_loop", kind="host_loop", model="1b", prompt=700, steps=16, K=7, n_max=4, policy=1, corrupt=0.15),
        # One verification forward whose logits the program reads (sampling, scoring): 7B at 2048 cached positions, six rows.
        dict(name="7b_step_logits", kind="step", model="7b", prompt=2040, width=6, corrupt=0.39),
        # The same on the 1.1B model, eight rows, an odd length.
        dict(name="1b_step_logits", kind="step", model="1b", prompt=509, width=8, corrupt=0.25),
        # A new document: the prompt's forward, then the first step's logits.  7B, and 1.1B at a ragged length.
        dict(name="7b_prefill", kind="prefill", model="7b", prompt=1536, width=1, corrupt=0.39),
        dict(name="1b_prefill", kind="prefill", model="1b", prompt=333, width=4, corrupt=0.25),
        # Eight independent sequences share one weight stream, each with its own tables and its own acceptance (13B width).
        dict(name="13b_batch8", kind="batch", model="13b", depth=10, batch=8, prompt=512, new=32, K=6, n_max=7, policy=0, corrupt=0.25),
        # Two candidates per step, on a prompt whose long contexts mislead.
        dict(name="1b_two_candidates", kind="generate", model="1b", prompt=600, new=64, K=5, n_max=5, policy=0, corrupt=0.0, candidates=2),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(("ngram", "generate", "generate", "generate", "host_loop", "step", "step", "prefill", "prefill", "batch"))
    opts = dict(K=rng.randint(1, 7), n_max=rng.randint(3, 7), policy=rng.randint(0, 1), corrupt=round(rng.uniform(0.1, 0.4), 3))
    if kind == "ngram":
        return dict(kind=kind, prompt=_log_int(rng, 16, 4096), rounds=_log_int(rng, 4, 64), **opts)
    model = rng.choice(("tiny", "1b", "1b", "7b", "7b"))
    if kind == "generate":
        c = dict(kind=kind, model=model, prompt=_log_int(rng, 16, 1536), new=_log_int(rng, 8, 128 if model != "7b" else 64), **opts)
        if rng.random() < 0.15:
            c["K"] = 0
        elif rng.random() < 0.25:
            c["candidates"] = 2
        return c
    if kind == "host_loop":
        return dict(kind=kind, model=model, prompt=_log_int(rng, 16, 1536), steps=_log_int(rng, 4, 16), **opts)
    if kind == "step":
        return dict(kind=kind, model=model, prompt=_log_int(rng, 32, 4096), width=rng.randint(1, 8), corrupt=opts["corrupt"])
    if kind == "prefill":
        return dict(kind=kind, model=model, prompt=_log_int(rng, 8, 3072), width=rng.randint(1, 8), corrupt=opts["corrupt"])
    model = rng.choice(("1b", "7b", "13b"))
    return dict(kind="batch", model=model, depth={"1b": 22, "7b": 8, "13b": 8}[model], batch=rng.randint(2, 8), prompt=_log_int(rng, 16, 768),
                new=_log_int(rng, 8, 48), **opts)


# ---- inputs ---------------------------------------------------------------------------------------------------------------
def _cycle(rng: np.random.Generator, S: int) -> np.ndarray:
    order = rng.permutation(S)
    pi = np.empty(S, dtype=np.int64)
    pi[order] = np.roll(order, -1)
    return pi


def _walk(pi: np.ndarray, t: int, n: int) -> np.ndarray:
    out = np.empty(n, dtype=np.int64)
    for i in range(n):
        out[i] = t
        t = pi[t]
    return out


def _prompt(rng: np.random.Generator, pi: np.ndarray, n: int, corrupt: float) -> np.ndarray:
    """The cycle with replaced tokens, closed by one of its early tokens, so that the continuation walks a stretch already shown."""
    S = len(pi)
    clean = _walk(pi, int(rng.integers(S)), max(n - 1, 1))
    out = clean.copy()
    first = min(8, n // 4)
    hit = rng.random(len(out)) < corrupt
    hit[:first + 1] = False
    out[hit] = rng.integers(0, S, int(hit.sum()))
    return np.append(out, clean[first])[-n:].astype(np.int32)


def _misleading_prompt(rng: np.random.Generator, pi: np.ndarray, n: int) -> np.ndarray:
    """A stretch of the cycle shown three times; at every ninth token d its successor is replaced in the first showing, and in the
    other two a token stands before d.  So what followed the longest context of d is wrong, what followed d itself is right."""
    S = len(pi)
    length = max(8, (n - 1) * 9 // 29)
    stretch = _walk(pi, int(rng.integers(S)), length)
    forks = set(range(4, length - 2, 9))
    stray = rng.integers(0, S, length)
    body: list[int] = []
    for showing in range(3):
        for i, tok in enumerate(stretch):
            if showing and i in forks:
                body.append(int(stray[i]))
            body.append(int(stray[i]) if not showing and i - 1 in forks else int(tok))
    body.append(int(stretch[0]))
    fill = rng.integers(0, S, max(0, n - len(body)))
    return np.concatenate([fill, np.asarray(body)])[-n:].astype(np.int32)


def _weights(s: SimpleNamespace, gen: torch.Generator, pi: np.ndarray, dtype: torch.dtype) -> list[torch.Tensor]:
    """Tensors in the order anpd_model_create takes them, on the GPU."""
    def mat(rows, cols, std):
        return torch.empty(rows, cols, dtype=dtype, device="cuda").normal_(0.0, std, generator=gen)

    def gain():
        return 1.0 + 0.05 * torch.randn(s.d_model, device="cuda", generator=gen)

    dq, dkv, d, f = s.n_q_heads * s.head_dim, s.n_kv_heads * s.head_dim, s.d_model, s.d_ffn
    spread = 0.08 / math.sqrt(2 * s.n_layers)            # what each half of a layer adds per dimension
    idx = torch.arange(s.S, device="cuda")
    w = [mat(s.vocab, d, 0.002)]
    w[0][idx, idx] += 1.0
    proj = 0.02 * math.sqrt(4096 / d)                    # q, k, gate, ... of about the same spread at every width
    for _ in range(s.n_layers):
        w += [gain(), mat(dq, d, proj), mat(dkv, d, proj), mat(dkv, d, proj), mat(d, dq, spread / math.sqrt(dq)),
              gain(), mat(f, d, proj), mat(f, d, proj), mat(d, f, spread / math.sqrt(f))]
    head = mat(s.vocab, d, 0.002)
    head[torch.from_numpy(pi).to("cuda"), idx] += 1.0
    return w + [gain(), head]


class State:
    """Handles and inputs of one program; the library's memory goes back when the state does."""

    def __init__(self, case: dict):
        self.case, self.m, self.kv, self.ctxs = case, None, None, []

    def close(self):
        for c in self.ctxs:
            A.anpd_ngram_destroy(c)
        if self.kv is not None:
            A.anpd_kv_destroy(self.kv)
        if self.m is not None:
            A.anpd_model_destroy(self.m)
        self.m, self.kv, self.ctxs = None, None, []

    def __del__(self):
        self.close()


def prepare(case: dict, seed: int) -> State:
    st = State(case)
    rng = np.random.default_rng(seed)
    kind, n, batch = case["kind"], case["prompt"], case.get("batch", 1)
    if kind == "ngram":
        pi = _cycle(rng, 4096)
        st.prompt = _prompt(rng, pi, n, case["corrupt"])
        follow = _prompt(rng, pi, case["rounds"] * 6 + 8, case["corrupt"])
        cuts = np.concatenate([[0], np.cumsum(rng.integers(1, 7, case["rounds"]))])
        st.updates = [follow[a:b].copy() for a, b in zip(cuts[:-1], cuts[1:])]
        st.ctxs = [A.anpd_ngram_create(2, case["n_max"], n + case["rounds"] * 6 + 16, case["policy"])]
        return st
    s = shape_of(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    pi = _cycle(rng, s.S)
    st.stream = torch.cuda.Stream()
    w = _weights(s, gen, pi, torch.float32 if case["model"] == "tiny" else torch.bfloat16)
    torch.cuda.synchronize()
    st.m = A.anpd_model_create(s, w, st.stream.cuda_stream)
    del w
    torch.cuda.empty_cache()                             # the library has its own copy
    st.vocab = s.vocab
    room = {"generate": case.get("new", 0), "batch": case.get("new", 0), "host_loop": 8 * case.get("steps", 0)}.get(kind, 8) + 24
    st.kv = A.anpd_kv_create(st.m, n + room, batch)
    if case.get("candidates", 1) == 2:
        A.anpd_kv_set_candidates(st.kv, 2)
        st.prompts = [_misleading_prompt(rng, pi, n)]
    else:
        st.prompts = [_prompt(rng, pi, n, case["corrupt"]) for _ in range(batch)]
    if kind in ("generate", "batch", "host_loop"):
        st.ctxs = [A.anpd_ngram_create(2, case["n_max"], n + room, case["policy"], st.stream.cuda_stream) for _ in range(batch)]
    if kind in ("step", "prefill"):
        st.rows = _walk(pi, int(pi[st.prompts[0][-1]]), case["width"]).astype(np.int32)      # the confirmed token and a draft
    if kind in ("step", "host_loop"):
        st.first = A.anpd_prefill(st.m, st.kv, st.prompts[0])
    return st


# ---- one pass -------------------------------------------------------------------------------------------------------------
def _counts(stats: dict) -> np.ndarray:
    return np.asarray([stats["steps"], stats["drafted"], stats["accepted"], stats["generated"], stats["alt_wins"], *stats["hist_accepted"]])


def run(st: State):
    c = st.case
    if c["kind"] == "ngram":
        ctx, K = st.ctxs[0], c["K"]
        drafts = np.full((c["rounds"] + 1, K), -1, dtype=np.int32)
        A.anpd_ngram_reset(ctx)
        A.anpd_ngram_update(ctx, st.prompt)
        d = A.anpd_ngram_draft(ctx, K)
        drafts[0, :len(d)] = d
        for i, new in enumerate(st.updates):
            A.anpd_ngram_update(ctx, new)
            d = A.anpd_ngram_draft(ctx, K)
            drafts[i + 1, :len(d)] = d
        return {"drafts": drafts}
    if c["kind"] == "generate":
        out, stats = A.anpd_generate(st.m, st.kv, st.ctxs[0], st.prompts[0], c["new"], c["K"])
        return {"tokens": out, "counts": _counts(stats)}
    if c["kind"] == "batch":
        out, stats = A.anpd_generate_batch(st.m, st.kv, st.ctxs, np.stack(st.prompts), c["new"], c["K"])
        return {"tokens": out, "counts": np.stack([_counts(s) for s in stats])}
    if c["kind"] == "step":
        logits = A.anpd_verify_logits(st.m, st.kv, int(st.rows[0]), st.rows[1:], st.vocab)
        return {"logits": logits}
    if c["kind"] == "prefill":
        A.anpd_kv_truncate(st.kv, 0, 0)
        first = A.anpd_prefill(st.m, st.kv, st.prompts[0])
        logits = A.anpd_verify_logits(st.m, st.kv, int(st.rows[0]), st.rows[1:], st.vocab)
        return {"first": first, "logits": logits}
    # host_loop: Algorithm 1 with the loop in the user's program
    ctx = st.ctxs[0]
    A.anpd_kv_truncate(st.kv, 0, c["prompt"])
    A.anpd_ngram_reset(ctx)
    A.anpd_ngram_update(ctx, np.append(st.prompts[0], st.first))
    last, tokens, accepted = st.first, [], []
    for _ in range(c["steps"]):
        draft = A.anpd_ngram_draft(ctx, c["K"])
        a, nxt = A.anpd_verify(st.m, st.kv, last, draft)
        new = draft[:a] + [nxt]
        A.anpd_ngram_update(ctx, new)
        tokens += new
        accepted.append(a)
        last = nxt
    return {"tokens": np.asarray(tokens + [-1] * (8 * c["steps"] - len(tokens))), "accepted": np.asarray(accepted)}


# ---- what a pass cannot do without ------------------------------------------------------------------------------------------
def _tokens_per_step(K: int, corrupt: float) -> float:
    q = (1.0 - corrupt) ** 2                             # a draft token is right where it and its precedent are intact
    return sum(q ** i for i in range(K + 1))


def work(case: dict) -> dict:
    kind, n, batch = case["kind"], case["prompt"], case.get("batch", 1)
    if kind == "ngram":                                  # each token: two 16-byte records per level; each draft token: one per level
        levels, tokens = case["n_max"] - 1, n + 3.5 * case["rounds"]
        return {"bytes": 4 * tokens + 32 * levels * tokens + 16 * levels * case["K"] * (case["rounds"] + 1), "flops": 0}
    s = shape_of(case)
    dq, dkv = s.n_q_heads * s.head_dim, s.n_kv_heads * s.head_dim
    layers = s.n_layers * (s.d_model * (2 * dq + 2 * dkv) + 3 * s.d_model * s.d_ffn)
    head = s.vocab * s.d_model
    kv_tok = 4.0 * s.n_layers * dkv                      # bf16 K and V of one position

    def step(rows, kv_len, logits):
        return {"bytes": 2.0 * (layers + head) + batch * kv_tok * (kv_len + rows) + 4.0 * batch * rows * s.vocab * logits,
                "flops": batch * rows * (2.0 * (layers + head) + 4.0 * s.n_layers * dq * kv_len)}

    prefill = {"bytes": 2.0 * (layers + head) + batch * kv_tok * n,
               "flops": batch * (2.0 * layers * n + 2.0 * s.n_layers * dq * n * n + 2.0 * head)}
    if kind == "step":
        return step(case["width"], n, 1)
    if kind == "prefill":
        one = step(case["width"], n, 1)
        return {k: prefill[k] + one[k] for k in one}
    if kind == "host_loop":
        one, steps = step(case["K"] + 1, n, 0), case["steps"]
        return {k: steps * one[k] for k in one}
    steps = math.ceil(case["new"] / _tokens_per_step(case["K"], case["corrupt"] or 0.3))
    one = step(case["K"] + 1, n + case["new"] / 2, 0)
    return {k: prefill[k] + steps * one[k] for k in one}


def tolerance(case: dict):
    # Tokens, drafts and counts are whole numbers, decided far from every tie.
    if case["kind"] not in ("step", "prefill"):
        return "exact"
    # Logits: bf16 weights and cache.  Four times what the same sums taken in another order show (the library's plain projections
    # against its tensor-core ones at 7B and 1.1B: 0.7e-3 to 1.0e-3, and 0.7e-2 to 1.2e-2 for the largest difference).
    return {"rel": 4e-3, "max": 5e-2}
