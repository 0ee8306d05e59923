"""GPU: steps with prompts — the whole-text build of the dynamic automaton and the static match of a long row —
against the oracle: every output, every state of the automata, and the decoding steps that go on from them."""
import random

import numpy as np
import pytest

import oracle
from _parity import assert_dynamic_automata_equal, assert_same, gpu_run, oracle_run

pytestmark = pytest.mark.gpu
VOCAB = 50_000


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    import paper_2411_10666_b200 as pkg
    pkg.lib()
    return pkg


def _text(kind, n, rng, corpus):
    if kind == "distinct":
        return rng.sample(range(VOCAB), n)
    if kind == "one":
        return [7] * n
    if kind == "periodic":
        u = [rng.randrange(50) for _ in range(rng.randint(2, 40))]
        x = (u * (n // len(u) + 1))[:n]
        x[n // 3] = 49_999
        return x
    if kind == "fibonacci":                                 # many suffix links per state
        a, b = [1], [1, 2]
        while len(b) < n:
            a, b = b, b + a
        return b[:n]
    if kind == "corpus":                                    # ends in a long passage of the corpus
        k = rng.randint(0, len(corpus) - n)
        x = corpus[k:k + n]
        return [rng.randrange(400)] * min(5, n) + x[min(5, n):]
    k = {"two": 2, "few": 30, "many": 3000, "copies": 400}[kind]
    x = [min(int(rng.expovariate(8.0 / k)), k - 1) for _ in range(n)]
    if kind == "copies":
        for _ in range(n // 60):
            m = rng.randint(5, 120)
            src, dst = rng.randrange(n), rng.randrange(n)
            m = min(m, n - src, n - dst)
            x[dst:dst + m] = x[src:src + m]
    return x


KEYS = ("draft_tokens", "draft_len", "match_len", "source", "state", "status")
KINDS = ("distinct", "one", "periodic", "fibonacci", "corpus", "two", "few", "many", "copies")


@pytest.mark.parametrize("n", [47, 48, 64, 65, 127, 128, 129, 700, 1025, 2048, 4096, 4097, 8192, 8193])
def test_prompt_builds_the_oracles_automaton(P, n):
    rng = random.Random(n)
    base = [rng.randrange(400) for _ in range(12_000)]
    corpus = base + base[2000:7000] + base[1000:9000]       # passages that occur once, twice and three times
    kinds = KINDS if n < 3000 else KINDS[1:5] + KINDS[-1:]
    B, L, more = len(kinds), 16, 3
    tail = [[rng.randrange(3) for _ in range(30)] for _ in range(B)]
    rows = np.array([_text(k, n, rng, corpus) + t for k, t in zip(kinds, tail)], dtype=np.int32)
    counts = np.full((more, B), 10, dtype=np.int32)
    steps = rows[:, n:].reshape(B, more, 10).transpose(1, 0, 2).copy()
    st = P.StaticSam.build(np.array(corpus, dtype=np.int32), VOCAB)
    ref, ob, _ = oracle_run(np.array(corpus, dtype=np.int32), VOCAB, rows[:, :n], steps, counts, L, n + 30, threads=8)
    for slab in (0,) if n > 2000 else (0, 4096):
        got, batch = gpu_run(P, st, VOCAB, rows[:, :n], steps, counts, L, n + 30, slab_bytes=slab)
        assert_same(got, ref, "n %d" % n)
        assert_dynamic_automata_equal(batch, ob, range(B), n + 30)


def test_mixed_step_with_prompts_short_rows_and_refused_slots(P):
    """One step in which slots take a prompt, go on from one, take a few tokens, take none or are refused."""
    import torch
    rng = random.Random(5)
    corpus = np.array([rng.randrange(300) for _ in range(6000)], dtype=np.int32)
    B, n, L = 9, 300, 8
    first = np.array([_text("copies", n, rng, []) for _ in range(B)], dtype=np.int32)
    second = np.array([_text("copies", n, rng, []) for _ in range(B)], dtype=np.int32)
    c1 = np.array([0, 300, 48, 47, 7, 120, 0, 300, 1], dtype=np.int32)
    c2 = np.array([300, 60, 5, 200, 300, 0, 49, 301, -1], dtype=np.int32)
    second[6, 20] = 300                                     # a token outside the vocabulary
    st = P.StaticSam.build(corpus, 300)
    S = oracle.Sam(corpus)
    ob = oracle.Batch(S, corpus, B, 300, 700)
    batch = P.Batch(st, B, 700, max_draft_len=L, max_host_stride=n)
    host = P.Batch(st, B, 700, max_draft_len=L, max_host_stride=n)
    keys = ("draft_tokens", "draft_len", "match_len", "source", "state", "status")
    for toks, cnt in ((first, c1), (second, c2)):
        ref = ob.step(toks, cnt, L, 1)
        got = batch.step(torch.from_numpy(toks).cuda(), torch.from_numpy(cnt).cuda(), L).cpu()
        o = [np.empty(s, dtype=np.int32) for s in ((B, L), (B,), (B, 2), (B,), (B, 2), (B,))]
        P.binding.sam_step_host(host.handle, toks, n, cnt, L, *o)
        for k, h in zip(keys, o):
            assert np.array_equal(got[k], getattr(ref, k)), k
            assert np.array_equal(h, getattr(ref, k)), k
    assert set(ref.status.tolist()) == {0, 3, 4}


@pytest.mark.parametrize("n", [60, 1000, 1100, 2100])
def test_many_prompts_at_once(P, n):
    """Batches that fill the GPU build with fewer registers and leave the static side to the step kernel."""
    rng = random.Random(n)
    base = [rng.randrange(400) for _ in range(12_000)]
    corpus = base + base[2000:7000]
    B, L = 300, 16
    rows = np.array([_text(KINDS[i % len(KINDS)], n, rng, corpus) + [rng.randrange(9) for _ in range(8)] for i in range(B)], dtype=np.int32)
    counts = np.full((1, B), 8, dtype=np.int32)
    st = P.StaticSam.build(np.array(corpus, dtype=np.int32), VOCAB)
    ref, ob, _ = oracle_run(np.array(corpus, dtype=np.int32), VOCAB, rows[:, :n], rows[None, :, n:].copy(), counts, L, n + 8, threads=8)
    got, batch = gpu_run(P, st, VOCAB, rows[:, :n], rows[None, :, n:].copy(), counts, L, n + 8)
    assert_same(got, ref)
    assert_dynamic_automata_equal(batch, ob, range(0, B, 37), n + 8)


@pytest.mark.parametrize("B,per_step", [(1, True), (296, True), (297, True), (297, False), (8193, True)])
def test_steps_in_one_launch(P, B, per_step):
    """sam_run_steps over each kernel's range: ragged counts, steps without tokens, slots that are refused on the way,
    rows of up to 47 tokens, with and without room for every step's outputs, with and without a static automaton."""
    import torch
    rng = np.random.default_rng(B)
    vocab, K, steps, L, msl = 60, 47, 5, 9, 150
    corpus = rng.integers(0, vocab, size=5000, dtype=np.int32)
    corpus[1000:2000] = corpus[:1000]
    text = rng.integers(0, vocab, size=(B, steps * K + 1), dtype=np.int32)
    text[:, 100:200] = corpus[900:1000]                     # long static matches
    text[::3, 30:60] = text[::3, :30]
    counts = np.where(rng.random((steps, B)) < 0.3, 0, rng.integers(0, K + 1, size=(steps, B))).astype(np.int32)
    toks = np.stack([text[:, i * K:(i + 1) * K] for i in range(steps)]).copy()
    if B > 8:
        counts[1, 3] = -2; counts[2, 5] = K + 1; toks[1, 7, 4] = vocab; counts[1, 7] = 9; toks[3, 8, 0] = -7; counts[3, 8] = 1
    keys = ("draft_tokens", "draft_len", "match_len", "source", "state", "status")
    for static in (True, False):
        st = P.StaticSam.build(corpus, vocab) if static else None
        S = oracle.Sam(corpus) if static else None
        ob = oracle.Batch(S, corpus if static else None, B, vocab, msl, 2, 2, 5)
        batch = P.Batch(st, B, msl, max_draft_len=L, l_bias=2, min_match=2, vocab=vocab, stop_token=5)
        for turn in range(2):                               # the second run goes on from the first
            ref = [ob.step(toks[i], counts[i], L, 8) for i in range(steps)]
            out = batch.run_steps(torch.from_numpy(toks).cuda(), torch.from_numpy(counts).cuda(), L, per_step=per_step).cpu()
            for k in keys:
                exp = np.stack([getattr(r, k) for r in ref]) if per_step else getattr(ref[-1], k)
                assert np.array_equal(out[k], exp), (static, turn, k, np.argwhere(out[k] != exp)[:3])
        assert_dynamic_automata_equal(batch, ob, [b for b in (0, 2, 3, 100) if b < B and ref[-1].status[b] == 0], msl)


@pytest.mark.parametrize("B,stride,L", [(1, 1, 1), (16, 47, 9), (18, 48, 9), (74, 11, 40), (75, 11, 40), (86, 11, 40), (87, 11, 41), (700, 12, 40), (1037, 7, 3)])
def test_host_steps_of_every_size(P, B, stride, L):
    """Host arrays at the edges of each way their bytes travel (in the launch, as pairs, fetched ahead, in place), pageable and
    page-locked, with refused slots among them."""
    import torch
    rng = np.random.default_rng(B * 100 + stride)
    vocab, steps = 40, 4
    msl = stride * steps
    corpus = rng.integers(0, vocab, size=3000, dtype=np.int32)
    st, S = P.StaticSam.build(corpus, vocab), oracle.Sam(corpus)
    toks = rng.integers(0, vocab, size=(steps, B, stride), dtype=np.int32)
    counts = rng.integers(0, stride + 1, size=(steps, B)).astype(np.int32)
    if B > 10:
        counts[1, 3] = -1; counts[2, 9] = stride + 1; toks[1, 5, 0] = vocab; counts[1, 5] = 1
    shapes = ((B, L), (B,), (B, 2), (B,), (B, 2), (B,))
    for pinned in (False, True):
        ob = oracle.Batch(S, corpus, B, vocab, msl)
        batch = P.Batch(st, B, msl, max_draft_len=L, max_host_stride=stride)
        out = [torch.empty(s, dtype=torch.int32) for s in shapes]
        tt, ct = torch.from_numpy(toks), torch.from_numpy(counts)
        if pinned:
            out, tt, ct = [o.pin_memory() for o in out], tt.pin_memory(), ct.pin_memory()
        for i in range(steps):
            ref = ob.step(toks[i], counts[i], L, 8)
            for o in out:
                o.fill_(-77)
            P.binding.sam_step_host(batch.handle, tt[i], stride, ct[i], L, *out)
            for o, k in zip(out, ("draft_tokens", "draft_len", "match_len", "source", "state", "status")):
                assert np.array_equal(o.numpy(), getattr(ref, k)), (pinned, i, k)


@pytest.mark.parametrize("B", [740, 741, 889, 1184, 1185])
def test_steps_at_the_edges_of_the_register_budgets(P, B):
    """One step kernel for each number of blocks an SM holds: plain and verified steps at the first and last batch of each."""
    import torch
    rng = np.random.default_rng(B)
    vocab, K, L, steps, msl = 25, 7, 6, 3, 60
    corpus = rng.integers(0, vocab, size=4000, dtype=np.int32)
    st, S = P.StaticSam.build(corpus, vocab), oracle.Sam(corpus)
    toks = rng.integers(0, vocab, size=(steps, B, K), dtype=np.int32)
    counts = rng.integers(0, K + 1, size=(steps, B)).astype(np.int32)
    ob, batch = oracle.Batch(S, corpus, B, vocab, msl), P.Batch(st, B, msl, max_draft_len=L)
    keys = ("draft_tokens", "draft_len", "match_len", "source", "state", "status")
    out = [P.StepOutputs(B, L, batch.device) for _ in range(2)]
    for i in range(steps):
        ref = ob.step(toks[i], counts[i], L, 8)
        batch.step(torch.from_numpy(toks[i]).cuda(), torch.from_numpy(counts[i]).cuda(), L, out[0])
        for k, v in out[0].cpu().items():
            assert np.array_equal(v, getattr(ref, k)), k
    dr, dl = out[0].draft_tokens.cpu().numpy(), out[0].draft_len.cpu().numpy()
    target = np.where(rng.random((B, L + 1)) < 0.8, np.concatenate([dr, dr[:, :1]], 1), 1).clip(0, vocab - 1).astype(np.int32)
    m = np.array([next((j for j in range(n) if dr[b, j] != target[b, j]), n) + 1 for b, n in enumerate(dl)], dtype=np.int32)
    P.binding.sam_step_verified(batch.handle, torch.from_numpy(target).cuda(), out[0].draft_tokens, out[0].draft_len, None, L, *out[1].tensors())
    ref = ob.step(target, m, L, 8)
    for k in keys:
        assert np.array_equal(getattr(out[1], k).cpu().numpy(), getattr(ref, k)), k


@pytest.mark.parametrize("B", [64, 400])
def test_prompts_beside_others_the_pool_cannot_hold(P, B):
    """Prompts the pool has room for are taken, whatever others that never fit ask for at the same time."""
    import torch
    rng = np.random.default_rng(B)
    vocab, n, L, fits = 2000, 1000, 8, (B // 3, B - 5)
    rows = rng.integers(0, 25, size=(B, n), dtype=np.int32)
    for b in fits:
        rows[b] = rng.permutation(vocab)[:n]                # one state a token, no edge blocks
    toks, counts = torch.from_numpy(rows).cuda(), torch.full((B,), n, dtype=torch.int32, device="cuda")
    counts[list(fits)] = n // 2

    def takes(b):
        one = P.Batch(None, 1, n, max_draft_len=L, vocab=vocab, slab_bytes=4096)
        assert one.step(toks[b:b + 1], counts[b:b + 1], L).cpu()["status"][0] == 0
        total, free = one.pool_info()
        return total - free

    pool = sum(takes(b) for b in fits)
    assert pool == 2 * (n // 2 * 32 // 4096 + 1) and min(takes(b) for b in (0, 1, B // 2, B - 1)) >= pool + 6    # (they differ by one or two)
    for turn in range(30):
        batch = P.Batch(None, B, n, max_draft_len=L, vocab=vocab, slab_bytes=4096, pool_slabs=pool)
        status = batch.step(toks, counts, L).cpu()["status"]
        assert np.flatnonzero(status == 0).tolist() == list(fits), (turn, np.flatnonzero(status == 0))
        assert batch.pool_info() == (pool, 0)
        batch.close()


@pytest.mark.parametrize("B", [64, 400])
def test_as_many_prompts_as_the_pool_holds(P, B):
    """Prompts of one text against a pool that holds half of them and a rest too small for one more: that many are taken, and
    they are the oracle's; the others fail without holding anything."""
    import torch
    rng = np.random.default_rng(B + 1)
    vocab, n, L, holds = 60, 700, 8, B // 2
    row = rng.integers(0, vocab, size=n, dtype=np.int32)
    toks = torch.from_numpy(np.tile(row, (B, 1))).cuda()
    counts = torch.full((B,), n, dtype=torch.int32, device="cuda")
    ref = oracle.Batch(None, None, 1, vocab, n).step(row[None], np.array([n], dtype=np.int32), L, 1)
    one = P.Batch(None, 1, n, max_draft_len=L, vocab=vocab, slab_bytes=4096)
    one.step(toks[:1], counts[:1], L)
    total, free = one.pool_info()
    takes = total - free
    assert takes > 4
    for turn in range(10):
        batch = P.Batch(None, B, n, max_draft_len=L, vocab=vocab, slab_bytes=4096, pool_slabs=holds * takes + takes - 1)
        out = batch.step(toks, counts, L).cpu()
        done = out["status"] == 0
        assert done.sum() == holds and (out["status"][~done] == 1).all()
        assert batch.pool_info() == (holds * takes + takes - 1, takes - 1)
        for k in ("draft_tokens", "draft_len", "match_len", "source", "state"):
            assert (out[k][done] == getattr(ref, k)[0]).all(), k
        batch.reset()
        assert batch.pool_info() == (holds * takes + takes - 1,) * 2
        batch.close()


@pytest.mark.parametrize("B,static", [(7, True), (296, True), (297, True), (297, False), (1300, True), (1700, False), (8300, True)])
@pytest.mark.parametrize("wide", [48, 129, 300])
def test_wide_rows_with_and_without_prompts(P, B, static, wide):
    """A server that keeps one row width: steps whose rows could hold prompts and do not, steps where a few slots change hands,
    refused rows among both, narrow rows and several steps in one call in between.  Every output of every step, and the
    automata at the end, at the edges of the kernels' ranges."""
    import torch
    rng = np.random.default_rng(B * 1000 + wide)
    vocab, L, msl = 50, 9, 900
    corpus = rng.integers(0, vocab, size=6000, dtype=np.int32)
    corpus[2000:3000] = corpus[:1000]
    st, S = (P.StaticSam.build(corpus, vocab), oracle.Sam(corpus)) if static else (None, None)
    ob = oracle.Batch(S, corpus if static else None, B, vocab, msl, 1, 2, 5)
    batch = P.Batch(st, B, msl, max_draft_len=L, l_bias=1, min_match=2, vocab=vocab, stop_token=5)

    def rows(width, counts):
        t = rng.integers(0, vocab, size=(B, width), dtype=np.int32)
        for b in np.flatnonzero(counts > 20):               # passages of the corpus, and repeats
            k = rng.integers(0, 5000)
            t[b, 10:20] = corpus[k:k + 10]
            if width > 60:
                t[b, 45:60] = t[b, 20:35]
        return t

    def compare(toks, counts, got):
        ref = ob.step(toks, counts, L, 8)
        for k in KEYS:
            assert np.array_equal(got[k], getattr(ref, k)), (k, np.argwhere(got[k] != getattr(ref, k))[:3])

    def step(toks, counts):
        compare(toks, counts, batch.step(torch.from_numpy(toks).cuda(), torch.from_numpy(counts).cuda(), L).cpu())

    few = lambda: rng.integers(0, 7, size=B).astype(np.int32)
    counts = np.where(rng.random(B) < 0.8, rng.integers(48, wide + 1, size=B), few()).astype(np.int32)
    toks = rows(wide, counts)
    counts[1], counts[2], toks[3, 20] = wide + 1, -1, vocab       # refused: too many, fewer than none, a token out of range
    counts[3] = wide
    step(toks, counts)
    for i in range(3):                                      # no prompts, rows that could hold them
        c = few()
        step(rows(wide, c), c)
    c = few()
    step(rows(16, c), c)
    gone = np.unique(rng.integers(0, B, size=max(2, B // 20))).astype(np.int32)
    batch.reset(gone)
    for b in gone:
        ob.reset(b)
    c = few()
    c[gone] = rng.integers(40, wide + 1, size=len(gone))
    toks = rows(wide, c)
    toks[gone[0], 30], c[gone[0]] = -4, wide                # a new slot's prompt is refused
    step(toks, c)
    many = np.stack([few() for _ in range(3)])
    toks = np.stack([rows(wide, c) for c in many])
    out = batch.run_steps(torch.from_numpy(toks).cuda(), torch.from_numpy(many).cuda(), L).cpu()
    for i in range(3):
        compare(toks[i], many[i], {k: out[k][i] for k in KEYS})
    ok = [b for b in list(range(0, B, max(1, B // 6))) + gone.tolist()[1:3] if out["status"][-1][b] == 0]
    assert_dynamic_automata_equal(batch, ob, ok, msl)


def test_host_steps_with_prompts_in_a_batch_that_lists_them(P):
    """Host arrays, more than two slots an SM: the completion flag is the last launch's, with prompts in every, in some and in no
    row of a wide step."""
    rng = np.random.default_rng(3)
    vocab, B, W, L, msl = 30, 400, 90, 7, 500
    corpus = rng.integers(0, vocab, size=4000, dtype=np.int32)
    st, S = P.StaticSam.build(corpus, vocab), oracle.Sam(corpus)
    ob, batch = oracle.Batch(S, corpus, B, vocab, msl), P.Batch(st, B, msl, max_draft_len=L, max_host_stride=W)
    out = [np.empty(s, dtype=np.int32) for s in ((B, L), (B,), (B, 2), (B,), (B, 2), (B,))]
    for i, share in enumerate((0.5, 0.0, 0.5, 0.0, 1.0)):
        toks = rng.integers(0, vocab, size=(B, W), dtype=np.int32)
        counts = np.where(rng.random(B) < share, rng.integers(48, W + 1, size=B), rng.integers(0, 5, size=B)).astype(np.int32)
        ref = ob.step(toks, counts, L, 8)
        P.binding.sam_step_host(batch.handle, toks, W, counts, L, *out)
        for k, v in zip(KEYS, out):
            assert np.array_equal(v, getattr(ref, k)), (i, k)


@pytest.mark.parametrize("B,stride,L", [(43, 8, 40), (44, 8, 40), (127, 100, 9), (128, 3, 9), (129, 3, 9)])
def test_host_steps_at_the_edge_of_the_pairs(P, B, stride, L):
    """Outputs of at most 2048 words come back as pairs, more behind the completion flag; rows of 100 tokens hold prompts."""
    test_host_steps_of_every_size(P, B, stride, L)


@pytest.mark.parametrize("B", [64, 400, 1700, 8200])
def test_steps_with_prompts_replayed_from_a_graph(P, B):
    """A reset, a step with prompts and two wide steps without, captured once and replayed on other inputs: nothing of one pass
    (marks, the list of prompts, which buffer holds the order) is left over for the next."""
    import torch
    rng = np.random.default_rng(B)
    vocab, W, L, msl = 40, 70, 8, 200
    corpus = rng.integers(0, vocab, size=4000, dtype=np.int32)
    st, S = P.StaticSam.build(corpus, vocab), oracle.Sam(corpus)
    batch = P.Batch(st, B, msl, max_draft_len=L)
    toks = torch.zeros(3, B, W, dtype=torch.int32, device="cuda")
    counts = torch.zeros(3, B, dtype=torch.int32, device="cuda")
    outs = [P.StepOutputs(B, L, "cuda") for _ in range(3)]

    def one_pass():
        batch.reset()
        for i in range(3):
            batch.step(toks[i], counts[i], L, outs[i])

    one_pass()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        one_pass()
    for share in (0.5, 0.0, 1.0, 0.1):
        t = rng.integers(0, vocab, size=(3, B, W), dtype=np.int32)
        c = rng.integers(0, 6, size=(3, B)).astype(np.int32)
        c[0] = np.where(rng.random(B) < share, rng.integers(48, W + 1, size=B), c[0])
        toks.copy_(torch.from_numpy(t)); counts.copy_(torch.from_numpy(c))
        graph.replay()
        torch.cuda.synchronize()
        ob = oracle.Batch(S, corpus, B, vocab, msl)
        for i in range(3):
            ref = ob.step(t[i], c[i], L, 8)
            for k, v in outs[i].cpu().items():
                assert np.array_equal(v, getattr(ref, k)), (share, i, k)


@pytest.mark.parametrize("B,n", [(148, 991), (149, 480), (149, 481), (149, 1025), (149, 2049), (2723, 105)])
def test_prompts_at_the_edges_of_the_build_blocks(P, B, n):
    """One and two builds an SM, and rows of as many tokens as the block has threads, one more, and several times as many."""
    rng = random.Random(B + n)
    base = [rng.randrange(400) for _ in range(12_000)]
    corpus = base + base[2000:7000]
    L = 16
    rows = np.array([_text(KINDS[i % len(KINDS)], n, rng, corpus) + [rng.randrange(9) for _ in range(8)] for i in range(B)], dtype=np.int32)
    counts = np.full((1, B), 8, dtype=np.int32)
    st = P.StaticSam.build(np.array(corpus, dtype=np.int32), VOCAB)
    ref, ob, _ = oracle_run(np.array(corpus, dtype=np.int32), VOCAB, rows[:, :n], rows[None, :, n:].copy(), counts, L, n + 8, threads=8)
    got, batch = gpu_run(P, st, VOCAB, rows[:, :n], rows[None, :, n:].copy(), counts, L, n + 8)
    assert_same(got, ref)
    assert_dynamic_automata_equal(batch, ob, range(0, B, 7), n + 8)


def _replayed(P, st, B, vocab, msl, toks, counts, L, **more):
    """The same steps replayed at once and one after the other: (outputs, outputs, batch, batch)."""
    import torch
    t, c = torch.from_numpy(toks).cuda(), torch.from_numpy(counts).cuda()
    once, each = (P.Batch(st, B, msl, max_draft_len=L, vocab=vocab, **more) for _ in range(2))
    a = once.run_steps(t, c, L, per_step=True).cpu()
    rows = [each.step(t[i], c[i], L).cpu() for i in range(len(toks))]
    return a, {k: np.stack([r[k] for r in rows]) for k in KEYS}, once, each


@pytest.mark.parametrize("B", [1, 7, 150])
@pytest.mark.parametrize("K,most", [(1, 1), (3, 3), (16, 16), (33, 33), (47, 47)])
def test_replayed_chunks_of_steps(P, B, K, most):
    """Steps of one token to more than a chunk holds, many without tokens, over texts of every kind: what a slot has at the end
    of each step is the oracle's, wherever chunks, runs and passages of the corpus begin and end."""
    rng = random.Random(100 * B + K)
    base = [rng.randrange(400) for _ in range(6000)]
    corpus = base + base[2000:4000] + base[1000:3000]
    steps = max(6, 200 // most)
    texts = np.array([_text(("corpus", "copies", "periodic", "few", "one", "many", "fibonacci")[b % 7], K * steps, rng, corpus) for b in range(B)], dtype=np.int32)
    r = np.random.default_rng(B + K)
    counts = np.where(r.random((steps, B)) < 0.25, 0, r.integers(0, most + 1, size=(steps, B))).astype(np.int32)
    if B > 1:
        counts[:, 1] = 0; counts[:, 2] = most               # a slot that takes nothing, one whose rows are full
    toks = np.zeros((steps, B, K), dtype=np.int32)
    for b in range(B):
        at = np.concatenate([[0], np.cumsum(counts[:, b])])
        for i in range(steps):
            toks[i, b, :counts[i, b]] = texts[b, at[i]:at[i + 1]]
    L, msl = 6, K * steps
    st = P.StaticSam.build(np.array(corpus, dtype=np.int32), VOCAB)
    ob = oracle.Batch(oracle.Sam(np.array(corpus, dtype=np.int32)), np.array(corpus, dtype=np.int32), B, VOCAB, msl)
    ref = [ob.step(toks[i], counts[i], L, 8) for i in range(steps)]
    got, each, once, _ = _replayed(P, st, B, VOCAB, msl, toks, counts, L)
    for k in KEYS:
        exp = np.stack([getattr(x, k) for x in ref])
        assert np.array_equal(got[k], exp), (k, np.argwhere(got[k] != exp)[:3])
        assert np.array_equal(each[k], exp), k
    assert_dynamic_automata_equal(once, ob, range(0, B, 5), msl)


@pytest.mark.parametrize("B", [1, 296, 297])
@pytest.mark.parametrize("steps,L", [(2, 128), (16, 128), (17, 128), (32, 33), (33, 33), (64, 32), (65, 32), (64, 1)])
def test_replays_of_few_steps_and_of_wide_ones(P, B, steps, L):
    """Up to 296 slots the rows are finished by the slot's own block as long as there are few, else by a launch of their own, as for
    more slots.  Steps of 16 and 17, 31 to 33 and 47 tokens side by side, where a chunk holds one step, two or a part, and slots
    refused at one of them: a token outside the vocabulary among the first 32 or behind them, a count, the capacity."""
    import torch
    K, vocab = 47, 300
    rng = np.random.default_rng(steps * 1000 + L + B)
    corpus = rng.integers(0, vocab, size=4000, dtype=np.int32)
    corpus[2000:3000] = corpus[:1000]
    counts = rng.choice([0, 1, 16, 17, 31, 32, 33, 47], size=(steps, B)).astype(np.int32)
    toks = rng.integers(0, vocab, size=(steps, B, K), dtype=np.int32)
    for i in range(steps):                                  # every second step goes on along the corpus
        if i % 2:
            at = rng.integers(0, 3900, size=B)
            toks[i] = corpus[at[:, None] + np.arange(K)]
    msl = max(int(counts.sum()), 1) if B == 1 else K * steps - 1
    if B > 10:
        mid = steps // 2
        counts[mid, :6] = (40, 40, 20, 33, K + 1, -1)
        toks[mid, 0, 39] = vocab; toks[mid, 1, 31] = -3; toks[mid, 2, 19] = vocab; toks[mid, 3, 32] = -1
        toks[:, 6] = 5; counts[:, 6] = 47                   # ... and slot 6 runs over the longest text there is
    st = P.StaticSam.build(corpus, vocab)
    ob = oracle.Batch(oracle.Sam(corpus), corpus, B, vocab, msl, 1, 2, 5)
    ref = [ob.step(toks[i], counts[i], L, 8) for i in range(steps)]
    assert B == 1 or ((ref[-1].status[:7] != 0).all() and (ref[-1].status[7:] == 0).any())
    t, c = torch.from_numpy(toks).cuda(), torch.from_numpy(counts).cuda()
    for per_step in (True, False):
        batch = P.Batch(st, B, msl, max_draft_len=L, l_bias=1, min_match=2, vocab=vocab, stop_token=5)
        got = batch.run_steps(t, c, L, per_step=per_step).cpu()
        for k in KEYS:
            exp = np.stack([getattr(r, k) for r in ref]) if per_step else getattr(ref[-1], k)
            assert np.array_equal(got[k], exp), (per_step, k, np.argwhere(got[k] != exp)[:3])
        assert_dynamic_automata_equal(batch, ob, [b for b in (0, 7, 100) if b < B and ref[-1].status[b] == 0], msl)


DUMP = ("n_tokens", "n_states", "n_edges", "length", "link", "min_endpos", "deg")


def _dump(batch, slot):
    d = batch.dump(slot, 4000, 8000)
    return {k: d[k].tolist() if hasattr(d[k], "tolist") else d[k] for k in DUMP}, sorted(zip(*(d["edge_" + k].tolist() for k in ("src", "tok", "tgt"))))


def test_replayed_steps_that_run_out_of_room(P):
    """A slot the pool has no slab left for fails at the same step, and is left as the step before left it, replayed or not."""
    rng = random.Random(3)
    B, K, steps, L, msl = 3, 11, 150, 4, 2000
    toks = np.zeros((steps, B, K), dtype=np.int32)
    toks[:, 0] = np.array(_text("copies", K * steps, rng, []), dtype=np.int32).reshape(steps, K)
    counts = np.zeros((steps, B), dtype=np.int32)
    counts[:, 0] = [rng.randint(0, K) for _ in range(steps)]
    for slabs in (2, 3, 6):
        got, each, once, one = _replayed(P, None, B, VOCAB, msl, toks, counts, L, pool_slabs=slabs, slab_bytes=8192)
        for k in KEYS:
            assert np.array_equal(got[k], each[k]), (slabs, k, np.argwhere(got[k] != each[k])[:3])
        assert (got["status"][-1, 0] == 1) and (got["status"][:, 1:] == 0).all()
        a, b = (x.dump(0, 4000, 8000) for x in (once, one))
        assert a["n_tokens"] == b["n_tokens"] and a["n_states"] == b["n_states"]
        assert _dump(once, 0) == _dump(one, 0)


@pytest.mark.parametrize("static", [False, True])
@pytest.mark.parametrize("kind,m,parts", [("distinct", 5, 1), ("distinct", 5, 2), ("distinct", 7, 1), ("distinct", 43, 1), ("one", 3, 1),
                                          ("fibonacci", 1, 1), ("copies", 1, 1), ("copies", 6, 2), ("corpus", 4, 1)])
def test_the_newest_state_of_a_replay_that_ran_out_of_room(P, kind, m, parts, static):
    """The pool ends exactly at a step's end (255 states: 51 steps of 5 new tokens, each token a state; the last also as the first
    step of a second launch) or inside a step: every record of the slot, the newest state's too, is that of the slot stepped one
    call at a time, and the steps before are the oracle's.  The pool holds garbage to begin with."""
    import torch
    rng = random.Random(m)
    L, msl, slabs, slab = 4, 1000, 2, 4096
    steps = 2 * 255 // m
    corpus = np.array([rng.randrange(400) for _ in range(3000)], dtype=np.int32)
    st = P.StaticSam.build(corpus, VOCAB) if static else None
    text = np.array(_text(kind, steps * m, rng, corpus.tolist()), dtype=np.int32)
    toks, counts = text.reshape(steps, 1, m), np.full((steps, 1), m, dtype=np.int32)
    t, c = torch.from_numpy(toks).cuda(), torch.from_numpy(counts).cuda()
    once, one = (P.Batch(st, 1, msl, max_draft_len=L, vocab=VOCAB, pool_slabs=slabs, slab_bytes=slab) for _ in range(2))
    for b in (once, one):
        b.workspace[-slabs * slab:] = 0xEE
    rows = [one.step(t[i], c[i], L).cpu() for i in range(steps)]
    each = {k: np.stack([r[k] for r in rows]) for k in KEYS}
    ok = int((each["status"][:, 0] == 0).sum())
    assert 0 < ok < steps and (each["status"][ok:] == 1).all()
    cuts = [0, ok, steps] if parts == 2 else [0, steps]
    outs = [once.run_steps(t[a:b].contiguous(), c[a:b].contiguous(), L, per_step=True).cpu() for a, b in zip(cuts, cuts[1:])]
    got = {k: np.concatenate([o[k] for o in outs]) for k in KEYS}
    ob = oracle.Batch(oracle.Sam(corpus) if static else None, corpus if static else None, 1, VOCAB, msl)
    for i in range(ok):
        ref = ob.step(toks[i], counts[i], L)
        for k in KEYS:
            assert np.array_equal(got[k][i], getattr(ref, k)) and np.array_equal(each[k][i], getattr(ref, k)), (i, k)
    for k in KEYS:
        assert np.array_equal(got[k][ok:], each[k][ok:]), k
    a, b = _dump(once, 0), _dump(one, 0)
    assert a == b
    assert a[0]["n_tokens"] == ok * m and ok * m in a[0]["length"]
    # exactly at a step's end: nothing of the next step has been made, so all of it is the oracle's
    if kind == "distinct" and m == 5:
        assert a[0]["n_states"] == 256
        assert_dynamic_automata_equal(once, ob, [0], msl)


def test_steps_before_the_one_whose_links_go_on_for_too_long(P, tmp_path):
    """In an automaton with a state whose suffix link leads to itself the walk's limit ends the step that meets it; the steps before
    it, in the same chunk of a replay too, are reported as they are one call at a time."""
    import torch
    path = str(tmp_path / "linked_to_itself.sam")
    st = P.StaticSam.build(np.array([1, 2, 3, 4, 5, 6, 7, 8, 9, 50, 5, 6, 7, 60], dtype=np.int32), 1000)
    st.save(path)
    words = np.fromfile(path, dtype=np.uint64)
    recs = words[16:16 + 4 * st.info.n_states].view(np.uint32).reshape(-1, 8)     # {len, link, first end position, ...} behind the header
    bad = int(np.flatnonzero((recs[:, 0] == 7) & (recs[:, 2] == 7))[0])           # the prefix of seven tokens
    recs[bad, 1] = bad
    total = 0xCBF29CE484222325
    for w in words[16:].tolist():
        total = (total ^ w) * 0x100000001B3 & 0xFFFFFFFFFFFFFFFF
    words[15] = total
    words.tofile(path)
    rows = [[1, 2], [3, 4, 5], [], [6, 7], [999], [1]]
    toks, counts = np.zeros((6, 1, 3), dtype=np.int32), np.array([[len(r)] for r in rows], dtype=np.int32)
    for i, r in enumerate(rows):
        toks[i, 0, :len(r)] = r
    got, each, _, _ = _replayed(P, P.StaticSam.load(path), 1, 1000, 64, toks, counts, 4)
    assert each["status"][:, 0].tolist() == [0, 0, 0, 0, 2, 2] and each["match_len"][3, 0, 0] == 7
    for k in KEYS:
        assert np.array_equal(got[k], each[k]), k


@pytest.mark.parametrize("record,slab", [((5, 1, 5, 1000, 0x7FFFFFFF, 16, 0, 0), None), ((5, 1, 5, 0xFFFFFFF0, 0, 16, 0, 0), None),
                                         ((5, 1, 5, 200, 95, 16, 0, 0), None), (None, 0x7FFFFFFF)])
def test_dumps_read_inside_the_pool(P, record, slab):
    """A record that names an edge block outside the pool (or one that is none) has no edges in a dump, a state slab outside it
    holds no states; the other states' are as they were."""
    import torch
    batch = P.Batch(None, 2, 100, max_draft_len=4, vocab=VOCAB, slab_bytes=4096, pool_slabs=3)
    toks = torch.tensor([[1, 2, 3, 4, 1, 2, 9, 9, 1, 5]] * 2, dtype=torch.int32, device="cuda")
    batch.step(toks, torch.tensor([10, 0], dtype=torch.int32, device="cuda"), 4)
    before = batch.dump(0, 100, 100)
    words = batch.workspace.view(torch.int32)
    pool = words[-3 * 1024:]
    state = 4
    at = int(words[64 + 16]) * 1024 + state * 8             # the slot's first slab, behind the pool's header and 16 control words
    assert pool[at].item() == before["length"][state] == 4
    if slab is None:
        pool[at:at + 8] = torch.tensor(np.array(record, dtype=np.uint32).view(np.int32), device="cuda")
    else:
        words[64 + 16] = slab
    after = batch.dump(0, 100, 100)
    edges = [[e for e in zip(*(d["edge_" + k].tolist() for k in ("src", "tok", "tgt"))) if e[0] == 0 or (slab is None and e[0] != state)] for d in (before, after)]
    assert after["n_states"] == before["n_states"] and after["n_edges"] == len(edges[1]) and edges[0] == edges[1]


@pytest.mark.parametrize("B", [64, 700, 1100, 1300])
def test_runs_of_new_tokens_with_a_known_one_behind(P, B):
    """Steps of r new tokens, a known one and what may follow it, for every r up to more than a warp holds: known by a solid
    transition of the root or not (a clone), the first token of the text, a token of the step itself."""
    import torch
    rng = random.Random(B)
    K, steps = 47, 4
    toks, counts = np.zeros((steps, B, K), dtype=np.int32), np.zeros((steps, B), dtype=np.int32)
    for b in range(B):
        fresh = iter(rng.sample(range(1000, VOCAB), 300))
        past = []
        for i in range(steps):
            row = [next(fresh) for _ in range(b % 42)]
            if past:
                row.append(past[0] if rng.random() < 0.2 else rng.choice(past))
            elif row:
                row.append(row[rng.randrange(len(row))])
            row += [rng.choice(past + row + [3, 4]) for _ in range(rng.randint(0, 3))]
            row = row[:K]
            past += row
            counts[i, b] = len(row)
            toks[i, b, :len(row)] = row
    L, msl = 5, K * steps
    ob = oracle.Batch(None, None, B, VOCAB, msl)
    batch = P.Batch(None, B, msl, max_draft_len=L, vocab=VOCAB)
    for i in range(steps):
        ref = ob.step(toks[i], counts[i], L, 8)
        got = batch.step(torch.from_numpy(toks[i]).cuda(), torch.from_numpy(counts[i]).cuda(), L).cpu()
        for k in KEYS:
            assert np.array_equal(got[k], getattr(ref, k)), (i, k)
    assert_dynamic_automata_equal(batch, ob, range(0, B, 13), msl)
