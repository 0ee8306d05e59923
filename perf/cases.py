"""The work whose speed is tracked: what a serving process has the library do, through its Python package.

A case is one pass over inputs that are in hand: a one-shot retrieval, a call for tree drafts, the prefill of a batch
of prompts, or a batch of requests served from the empty batch through every decoding step.  A batch's automata grow
with every token, so a pass that decodes begins by resetting the batch and feeding the prompts, as a server does when
it takes a new batch in; the same state can then be passed over again.

The static automaton is what a server builds once and keeps: it is made from a corpus that depends on the case alone.
Prompts, generated text, accepted-token counts and the slots that change hands depend on the seed.  Texts follow the
repository's workload recipes (Zipf-distributed token ids, in some of them rotated by the two tokens before; verbatim
copies of spans of the corpus and of the own text), drawn on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2411_10666_b200 as P

# tokens: corpus length; zipf, markov: the token model; copies, span: share of positions inside copied spans, and
# the spans' lengths; rows: the texts the corpus is made of, all drawn side by side; eos: joins them, ends a draft;
# topk: successors kept for tree drafts
CORPORA = {
    "small": dict(tokens=100_000, vocab=32000, zipf=1.1, markov=False, copies=0.30, span=(8, 64), rows=100),
    "topic": dict(tokens=1_000_000, vocab=32000, zipf=1.1, markov=False, copies=0.0, span=(8, 64), rows=1000),
    "docs": dict(tokens=4_000_000, vocab=32000, zipf=1.1, markov=True, copies=0.25, span=(8, 128), rows=8000, eos=31999, topk=4),
    "wide": dict(tokens=8_000_000, vocab=128256, zipf=1.05, markov=True, copies=0.25, span=(8, 256), rows=8000),
    "frequent": dict(tokens=4_000_000, vocab=128256, zipf=1.05, markov=False, copies=0.20, span=(16, 256), rows=4000),
}
DEVICE = 0
_shared = {}            # corpus name -> (automaton, corpus on the device, token model): one of each per process


def listed():
    return [
        # one request's text so far, looked up by a hook that may not allocate: the smallest call there is
        dict(name="retrieve_1x300", kind="retrieve", corpus="small", batch=1, prompt=300, draft=16),
        # the same for a handful of requests, near what the built-in scratch array holds
        dict(name="retrieve_16x1000", kind="retrieve", corpus="docs", batch=16, prompt=1000, draft=32),
        # tree drafts for a batch in mid-generation
        dict(name="tree_64x40", kind="tree", corpus="docs", batch=64, nodes=40, topk=4),
        # a batch of prompts, the sequences' first step
        dict(name="prefill_64x1024", kind="prefill", corpus="docs", batch=64, prompt=1024, draft=32, copies=0.35, from_corpus=0.5),
        # one user's long context
        dict(name="prefill_1x8191", kind="prefill", corpus="frequent", batch=1, prompt=8191, draft=32, copies=0.30, from_corpus=0.5),
        # four sequences, tokens kept on the host: the smallest decoding step, end to end
        dict(name="host_4", kind="decode", api="host", corpus="small", batch=4, prompt=256, steps=192, accept=4, p=0.0,
             draft=16, copies=0.40, from_corpus=0.5),
        # prompt-copying generation over long prompts, tokens kept on the host: nearly all drafts come from the own text
        dict(name="host_1000", kind="decode", api="host", corpus="topic", batch=1000, prompt=1500, steps=192, accept=12, p=0.25,
             draft=40, copies=0.60, from_corpus=0.0, plain_prompt=True),
        # one call per step from Python with everything on the device
        dict(name="step_64", kind="decode", api="step", corpus="docs", batch=64, prompt=1024, steps=256, accept=8, p=0.4,
             draft=32, copies=0.35, from_corpus=0.5),
        # the closed loop: the target's tokens verified and fed back in the step's own launch
        dict(name="verified_256", kind="verified", corpus="frequent", batch=256, prompt=1024, steps=192, draft=32,
             copies=0.30, from_corpus=0.5),
        # continuous batching: slots change hands all the time, an auxiliary drafter fills in where the match is short
        dict(name="serve_200", kind="serve", corpus="docs", batch=200, prompt=700, steps=64, accept=8, p=0.4, draft=32,
             copies=0.35, from_corpus=0.5, arrivals=8),
        # a large batch of recorded requests replayed step after step
        dict(name="replay_4096", kind="decode", api="replay", corpus="wide", batch=4096, prompt=1024, steps=192, accept=16, p=0.3,
             draft=32, copies=0.40, from_corpus=0.5),
        # as many sequences as a GPU of this size is asked to hold
        dict(name="replay_16384", kind="decode", api="replay", corpus="wide", batch=16384, prompt=300, steps=96, accept=16, p=0.3,
             draft=32, copies=0.40, from_corpus=0.5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["retrieve", "tree", "prefill", "decode", "decode", "decode", "verified", "serve"])
    copies, from_corpus = round(rng.uniform(0.2, 0.6), 2), rng.choice([0.0, 0.5, 0.5])
    draft = rng.choice([16, 32, 32, 40])
    text = dict(copies=copies, from_corpus=from_corpus)
    corpus = rng.choice(["small", "topic", "docs", "wide", "frequent", "none"])
    if kind == "retrieve":
        batch = _log(rng, 1, 16)
        return dict(kind=kind, corpus=corpus, batch=batch, prompt=_log(rng, 50, 1000), draft=draft)
    if kind == "tree":
        return dict(kind=kind, corpus="docs", batch=_log(rng, 1, 4096), nodes=_log(rng, 8, 100), topk=rng.choice([1, 2, 3, 4]))
    if kind == "prefill":
        batch = _log(rng, 1, 4096)
        return dict(kind=kind, corpus=corpus, batch=batch, prompt=_log(rng, 100, min(8191, 2_000_000 // batch)), draft=draft, **text)
    accept = rng.choice([4, 8, 12, 16])
    p = rng.choice([0.25, 0.3, 0.4])
    if kind == "verified":
        batch = _log(rng, 1, 1000)
        return dict(kind=kind, corpus=corpus, batch=batch, prompt=_log(rng, 100, 2000), steps=_log(rng, 32, 192), draft=draft, **text)
    if kind == "serve":
        batch = _log(rng, 8, 1000)
        return dict(kind=kind, corpus=corpus, batch=batch, prompt=_log(rng, 100, 1500), steps=_log(rng, 32, 96), accept=accept, p=p,
                    draft=draft, arrivals=max(1, batch // rng.choice([16, 32])), **text)
    api = rng.choice(["host", "step", "replay"])
    batch = _log(rng, 1, 4096 if api == "host" else 12000)
    longest = min(2000, 4_000_000 // batch)
    return dict(kind=kind, api=api, corpus=corpus, batch=batch, prompt=_log(rng, 50, longest), steps=_log(rng, 32, 192 if batch <= 4096 else 96),
                accept=accept, p=p, draft=draft, **text)


# ---------------------------------------------------------------------------------------------------- texts
def _generator(*key):
    return torch.Generator(device=DEVICE).manual_seed(hash(key) & 0x7FFFFFFFFFFF)


class _Tokens:
    """Zipf-distributed token ids; with `markov`, each pair of tokens before has a ranking of its own."""

    def __init__(self, vocab, zipf, markov, seed):
        w = torch.arange(1, vocab + 1, dtype=torch.float64, device=DEVICE).pow_(-zipf)
        self.cdf = torch.cumsum(w, 0) / w.sum()
        self.perm = torch.randperm(vocab, generator=_generator(seed, 1), device=DEVICE)
        self.vocab, self.markov = vocab, markov

    def texts(self, rows, length, g, copies, span, corpus=None, from_corpus=0.0, plain=0, own_limit=0, any_row=False):
        """int32 [rows, length]: fresh tokens, and spans copied from `corpus` (share `from_corpus` of the spans) or from
        the own text (with any_row: from all rows' texts); the first `plain` positions hold no copies; with own_limit,
        own-text copies read the first own_limit positions only."""
        n, dev = length, DEVICE
        rank = torch.searchsorted(self.cdf, torch.rand(n, rows, generator=g, device=dev, dtype=torch.float64)).clamp_(max=self.vocab - 1)
        at = torch.arange(n, device=dev)[:, None]
        mean = 0.5 * (span[0] + span[1])
        q = copies / (copies + mean * (1.0 - copies)) if copies > 0 else 0.0
        start = (torch.rand(n, rows, generator=g, device=dev) < q) & (at >= max(1, plain))
        last = torch.where(start, at, -1).cummax(0).values                      # where the latest span began
        length_of = torch.randint(span[0], span[1] + 1, (n, rows), generator=g, device=dev)
        u = torch.rand(n, rows, generator=g, device=dev, dtype=torch.float64)
        outer = torch.rand(n, rows, generator=g, device=dev) < (from_corpus if corpus is not None else 0.0)
        row = torch.randint(0, rows, (n, rows), generator=g, device=dev) if any_row else torch.arange(rows, device=dev).expand(n, rows)
        k = last.clamp(min=0)
        inside = (last >= 0) & (at - k < length_of.gather(0, k))
        outer, u, row = outer.gather(0, k), u.gather(0, k), row.gather(0, k)
        limit = k.clamp(max=own_limit) if own_limit else k
        src = (u * limit).long() + (at - k)                                     # always before `at`
        if own_limit:
            inside &= outer | (src < own_limit)
        far = corpus[((u * corpus.numel()).long() + (at - k)) % corpus.numel()].long() if corpus is not None else None
        out = torch.empty(n, rows, dtype=torch.int64, device=dev)
        flat = out.view(-1)
        cell = src.clamp(min=0) * rows + row
        fresh = self.perm[rank]
        for i in range(n):
            new = fresh[i]
            if self.markov and i >= 2:
                mix = out[i - 2] * 1_000_003 + out[i - 1] * 7_919
                new = self.perm[(rank[i] + (mix ^ (mix >> 11))) % self.vocab]
            if i > 0 and q > 0:
                old = flat[cell[i]]
                if far is not None:
                    old = torch.where(outer[i], far[i], old)
                new = torch.where(inside[i], old, new)
            out[i] = new
        return out.t().to(torch.int32).contiguous()


def _static(name):
    """(automaton or None, corpus or None, token model) of a corpus; built once per process and kept, as a server does."""
    if name not in _shared:
        if name == "none":                                                      # no retrieval corpus: the own text is all there is
            _shared[name] = (None, None, _Tokens(32000, 1.1, False, 77))
            return _shared[name]
        c = CORPORA[name]
        model = _Tokens(c["vocab"], c["zipf"], c["markov"], 11)
        g = _generator(len(name), c["tokens"])
        text = model.texts(c["rows"], c["tokens"] // c["rows"], g, c["copies"], c["span"], any_row=True)
        if "eos" in c:
            text[text == c["eos"]] = 0
            text[:, -1] = c["eos"]
        text = text.view(-1)
        static = P.StaticSam.build(text.cpu().numpy(), c["vocab"], device=DEVICE, tree_topk=c.get("topk", 0))
        if name == "topic":                                                     # requests about something else than the corpus
            model = _Tokens(c["vocab"], c["zipf"], c["markov"], 12)
        _shared[name] = (static, text, model)
    return _shared[name]


def _texts(case, seed, rows, length):
    static, corpus, model = _static(case["corpus"])
    c = CORPORA.get(case["corpus"], CORPORA["small"])
    prompt = case.get("prompt", length)
    plain = prompt if case.get("plain_prompt") else 0
    return model.texts(rows, length, _generator(seed, 2), case.get("copies", 0.35), c["span"], corpus=corpus,
                       from_corpus=case.get("from_corpus", 0.5), plain=plain, own_limit=prompt if plain else 0)


def _counts(case, seed, rows):
    """Accepted tokens per step, int32 [steps, rows]: uniform on 1..accept with p = 0, else geometric(p) cut at accept."""
    g, K = _generator(seed, 3), case["accept"]
    u = torch.rand(case["steps"], rows, generator=g, device=DEVICE, dtype=torch.float64)
    n = u * K + 1 if case["p"] == 0 else torch.log1p(-u) / math.log1p(-case["p"]) + 1
    return n.floor().clamp_(1, K).to(torch.int32)


def _rows_of_steps(texts, first, counts, width):
    """int32 [steps, rows, width]: step i's tokens of every row, -1 from its count on; first[row]: where step 0 begins."""
    begin = torch.cumsum(counts.long(), 0) - counts + first
    j = torch.arange(width, device=DEVICE)
    tokens = torch.stack([texts.gather(1, (b[:, None] + j).clamp_(max=texts.shape[1] - 1)) for b in begin])
    return torch.where(j < counts[:, :, None], tokens, -1).contiguous()


# ---------------------------------------------------------------------------------------------------- states
class _State:
    pass


def _steps_of(out, n):
    """The n per-step views of outputs that keep every step."""
    steps = []
    for i in range(n):
        o = P.StepOutputs.__new__(P.StepOutputs)
        for name in ("draft_tokens", "draft_len", "match_len", "source", "state", "status"):
            setattr(o, name, getattr(out, name)[i])
        steps.append(o)
    return steps


def _batch(case, static, max_seq_len, **more):
    c = CORPORA.get(case["corpus"], {})
    return P.Batch(static, case["batch"], max_seq_len, max_draft_len=case["draft"], vocab=0 if static else 32000,
                   device=DEVICE, stop_token=c.get("eos", -1), **more)


def prepare(case, seed):
    torch.cuda.set_device(DEVICE)
    s = _State()
    s.case = case
    static, _, _ = s.shared = _static(case["corpus"])
    globals()["_prepare_" + case["kind"]](s, case, seed, static)
    return s


def _prepare_retrieve(s, case, seed, static):
    B, n = case["batch"], case["prompt"]
    g = _generator(seed, 4)
    s.tokens = _texts(case, seed, B, n)
    s.counts = torch.randint((n + 1) // 2, n + 1, (B,), generator=g, device=DEVICE, dtype=torch.int32)   # ragged
    s.counts[0] = n
    s.out = P.StepOutputs(B, case["draft"], s.tokens.device)


def _prepare_tree(s, case, seed, static):
    # the static states that sequences are in after reading some text
    B = case["batch"]
    texts = _texts(case, seed, B, 48)
    batch = P.Batch(static, B, 64, max_draft_len=16)
    out = batch.step(texts, torch.full((B,), 48, dtype=torch.int32, device=DEVICE), 16)
    s.states, s.starts = out.state[:, 0].contiguous(), texts[:, -1].contiguous()
    batch.close()
    s.tokens = torch.empty(B, case["nodes"], dtype=torch.int32, device=DEVICE)
    s.parents = torch.empty_like(s.tokens)
    s.probs = torch.empty(B, case["nodes"], dtype=torch.float32, device=DEVICE)
    s.sizes = torch.empty(B, dtype=torch.int32, device=DEVICE)


def _prepare_prefill(s, case, seed, static):
    B, n = case["batch"], case["prompt"]
    s.prompts = _texts(case, seed, B, n)
    s.full = torch.full((B,), n, dtype=torch.int32, device=DEVICE)
    s.batch = _batch(case, static, n + 1024)
    s.out = P.StepOutputs(B, case["draft"], s.prompts.device)


def _prepare_decode(s, case, seed, static):
    B, n, steps = case["batch"], case["prompt"], case["steps"]
    counts = _counts(case, seed, B)
    longest = n + int(counts.sum(0).max())
    texts = _texts(case, seed, B, longest)
    s.prompts = texts[:, :n].contiguous()
    s.full = torch.full((B,), n, dtype=torch.int32, device=DEVICE)
    s.tokens, s.counts = _rows_of_steps(texts, n, counts, case["accept"]), counts.contiguous()
    s.batch = _batch(case, static, longest, max_host_stride=max(32, case["accept"]))
    L = case["draft"]
    if case["api"] == "host":
        # the arrays a server on the host keeps: page-locked, the outputs in one block with a view for each
        s.tokens = s.tokens.cpu().pin_memory()
        s.counts = s.counts.cpu().pin_memory()
        s.block = torch.empty(B * (L + 7), dtype=torch.int32).pin_memory()
        at, views = 0, []
        for shape in ((B, L), (B,), (B, 2), (B,), (B, 2), (B,)):
            size = int(np.prod(shape))
            views.append(s.block[at:at + size].view(shape))
            at += size
        s.kept = np.empty((steps, B * (L + 7)), dtype=np.int32)
        s.block_np = s.block.numpy()
        s.call = P.binding.sam_step_host_prepared(s.batch.handle, case["accept"], L, *views)
        s.ins = [(t, c) for t, c in zip(s.tokens, s.counts)]
        s.first = P.StepOutputs(B, L, s.prompts.device)
    else:
        s.out = P.StepOutputs(B, L, s.prompts.device, steps)
        s.first = P.StepOutputs(B, L, s.prompts.device)
        s.ins = list(zip(s.tokens, s.counts, _steps_of(s.out, steps))) if case["api"] == "step" else None


def _prepare_verified(s, case, seed, static):
    # The target model's tokens are those of the sequence's own continuation.  The loop is deterministic, so one pass
    # with the target played by index arithmetic records the rows the target hands over at every step.
    B, n, steps, L = case["batch"], case["prompt"], case["steps"], case["draft"]
    longest = n + 4 * steps + 2 * (L + 1)
    texts = _texts(case, seed, B, longest)
    s.prompts = texts[:, :n].contiguous()
    s.full = torch.full((B,), n, dtype=torch.int32, device=DEVICE)
    s.batch = _batch(case, static, longest)
    s.out = P.StepOutputs(B, L, s.prompts.device, steps + 1)
    s.steps = _steps_of(s.out, steps + 1)
    s.counts = torch.empty(steps, B, dtype=torch.int32, device=DEVICE)
    s.accepted = torch.empty_like(s.counts)
    s.caps = torch.empty_like(s.counts)
    s.targets = torch.empty(steps, B, L + 1, dtype=torch.int32, device=DEVICE)
    s.batch.step(s.prompts, s.full, L, s.steps[0])
    at, j = torch.full((B,), n, dtype=torch.int64, device=DEVICE), torch.arange(L + 1, device=DEVICE)
    for i in range(steps):
        s.targets[i] = texts.gather(1, (at[:, None] + j).clamp_(max=longest - 1))
        s.caps[i] = longest - at
        _verified_step(s, i, L)
        at += s.counts[i]


def _verified_step(s, i, L):
    P.binding.sam_step_verified(s.batch.handle, s.targets[i], s.steps[i].draft_tokens, s.steps[i].draft_len, s.caps[i], L,
                                *s.steps[i + 1].tensors(), counts_out=s.counts[i], accepted_out=s.accepted[i])


def _prepare_serve(s, case, seed, static):
    B, n, steps, L, K = case["batch"], case["prompt"], case["steps"], case["draft"], case["accept"]
    counts = _counts(case, seed, B)
    longest = n + int(counts.sum(0).max())
    texts = _texts(case, seed, B, longest)
    g = _generator(seed, 5)
    who = torch.rand(steps, B, generator=g, device=DEVICE).argsort(1)[:, :case["arrivals"]]
    new_prompts = _texts(case, seed + 1_000_003, steps * case["arrivals"], n).view(steps, case["arrivals"], n)
    lengths = torch.randint((n + 1) // 2, n + 1, (steps, case["arrivals"]), generator=g, device=DEVICE, dtype=torch.int32)
    s.prompts = texts[:, :n].contiguous()
    s.full = torch.full((B,), n, dtype=torch.int32, device=DEVICE)
    tokens = _rows_of_steps(texts, n, counts, K)
    s.ins = []
    s.out = P.StepOutputs(B, L, texts.device, steps)
    s.aux = torch.randint(0, 32000, (steps, B, L), generator=g, device=DEVICE, dtype=torch.int32)
    s.aux_len = torch.randint(0, L + 1, (steps, B), generator=g, device=DEVICE, dtype=torch.int32)
    slots = who.cpu().numpy().astype(np.int32)
    for i, out in enumerate(_steps_of(s.out, steps)):
        if i % 4 == 0:                                                          # every fourth step some slots change hands
            wide = torch.full((B, max(n, K)), -1, dtype=torch.int32, device=DEVICE)
            wide[:, :K] = tokens[i]
            wide[who[i]] = -1
            wide[who[i], :n] = new_prompts[i]
            count = counts[i].clone()
            count[who[i]] = lengths[i]
            s.ins.append((slots[i], wide, count, out, s.aux[i], s.aux_len[i]))
        else:
            s.ins.append((None, tokens[i], counts[i].contiguous(), out, s.aux[i], s.aux_len[i]))
    s.batch = _batch(case, static, longest, l_bias=5, min_match=5)
    s.first = P.StepOutputs(B, L, texts.device)


# ---------------------------------------------------------------------------------------------------- passes
def run(s):
    return globals()["_run_" + s.case["kind"]](s, s.case)


def _outputs(o):
    return dict(draft_tokens=o.draft_tokens, draft_len=o.draft_len, match_len=o.match_len, source=o.source, state=o.state, status=o.status)


def _run_retrieve(s, case):
    static = s.shared[0]
    P.binding.sam_retrieve_noalloc(static.handle if static else None, 32000, s.tokens, s.counts, case["draft"], 0, 1, *s.out.tensors())
    return _outputs(s.out)


def _run_tree(s, case):
    P.binding.sam_tree_draft(s.shared[0].handle, s.states, s.starts, case["nodes"], case["topk"], s.tokens, s.parents, s.probs, s.sizes)
    return dict(tokens=s.tokens, parents=s.parents, probs=s.probs, sizes=s.sizes)


def _run_prefill(s, case):
    s.batch.reset()
    return _outputs(s.batch.step(s.prompts, s.full, case["draft"], s.out))


def _run_decode(s, case):
    L = case["draft"]
    s.batch.reset()
    s.batch.step(s.prompts, s.full, L, s.first)
    if case["api"] == "host":
        for i, (tokens, counts) in enumerate(s.ins):
            s.call(tokens, counts)
            s.kept[i] = s.block_np
        return dict(first=_outputs(s.first), kept=s.kept)
    if case["api"] == "step":
        for tokens, counts, out in s.ins:
            s.batch.step(tokens, counts, L, out)
    else:
        s.batch.run_steps(s.tokens, s.counts, L, True, s.out)
    return dict(first=_outputs(s.first), steps=_outputs(s.out))


def _run_verified(s, case):
    L = case["draft"]
    s.batch.reset()
    s.batch.step(s.prompts, s.full, L, s.steps[0])
    for i in range(case["steps"]):
        _verified_step(s, i, L)
    return dict(steps=_outputs(s.out), counts=s.counts, accepted=s.accepted)


def _run_serve(s, case):
    L = case["draft"]
    s.batch.reset()
    s.batch.step(s.prompts, s.full, L, s.first)
    for slots, tokens, counts, out, aux, aux_len in s.ins:
        if slots is not None:
            s.batch.reset(slots)
        s.batch.step(tokens, counts, L, out)
        P.binding.sam_select_auxiliary(out.draft_tokens, out.draft_len, out.source, aux, aux_len)
    return dict(first=_outputs(s.first), steps=_outputs(s.out))


def work(case):
    """Bytes only, no arithmetic to speak of: tokens and counts in, outputs out, and per token one state of the corpus
    automaton read and one state (32 bytes), one position of the text and one transition (8) of the own automaton written."""
    if case["kind"] == "tree":
        # per node: its token, parent and probability written, its record, frequency and one candidate entry read
        return {"bytes": case["batch"] * (12 + case["nodes"] * (12 + 32 + 4 + 8 * case["topk"])), "flops": 2 * case["batch"] * case["nodes"] * case["topk"]}
    B, steps = case["batch"], case.get("steps", 0)
    p = case.get("p", 0)
    K = case.get("accept", 0)
    mean = (K + 1) / 2 if p == 0 else (1 - (1 - p) ** K) / p
    if case["kind"] == "verified":
        mean = 1.5
    tokens = B * (case["prompt"] * (0.75 if case["kind"] == "retrieve" else 1.0) + mean * steps)
    if case["kind"] == "serve":
        tokens += steps / 4 * case["arrivals"] * 0.75 * case["prompt"]
    per_token = 4 + (32 if case["corpus"] != "none" else 0) + 32 + 4 + 8
    return {"bytes": tokens * per_token + (steps + 1) * B * 4 * (1 + case["draft"] + 7), "flops": 0}


def tolerance(case):
    return "exact"              # whole numbers, and probabilities whose rounding is part of the interface
