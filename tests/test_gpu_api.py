"""GPU tests of the boundary's conventions: per-slot status codes, freezing, reset and slab reuse,
count 0, the host-array step, image save/load, pool exhaustion.  Expected values come from the
oracle or are stated outright; nothing here expects a fault."""
import os
import random

import numpy as np
import pytest

import oracle
import workloads as W
from _parity import KEYS, assert_dynamic_automata_equal, assert_same, gpu_run, oracle_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available()
    import paper_2411_10666_b200 as pkg
    pkg.lib()
    return pkg


def _t(a, dev):
    import torch
    return torch.from_numpy(np.ascontiguousarray(np.asarray(a, dtype=np.int32))).to(dev)


def test_status_codes_freeze_and_match_oracle(P):
    vocab, msl, L = 10, 6, 4
    steps = [
        ([[1, 2, 3], [1, 10, 0], [1, 2, 3], [1, 2, 3]], [3, 2, 4, 3]),     # ok, bad token, bad count, ok
        ([[1, 2, 1], [1, 1, 1], [1, 1, 1], [5, 0, 0]], [3, 1, 1, 1]),      # ok (6 tokens), frozen, frozen, ok
        ([[1, 0, 0], [1, 1, 1], [1, 1, 1], [5, 0, 0]], [1, 0, -1, 0]),     # capacity, frozen, frozen, count 0
    ]
    nt = np.array([s[0] for s in steps], dtype=np.int32)
    ct = np.array([s[1] for s in steps], dtype=np.int32)
    empty = np.zeros((4, 0), np.int32)
    ref, _, _ = oracle_run(None, vocab, empty, nt, ct, L, msl)
    got, batch = gpu_run(P, None, vocab, empty, nt, ct, L, msl)
    assert_same(got, ref)
    assert got["status"].tolist() == [[0, 3, 4, 0], [0, 3, 4, 0], [1, 3, 4, 0]]
    assert (got["draft_tokens"][2, :3] == -1).all() and (got["draft_len"][2, :3] == 0).all()
    # the failed step changed nothing: slot 0 still holds 6 tokens
    assert batch.dump(0, 16, 32)["n_tokens"] == 6


def test_argument_errors_launch_nothing(P):
    import torch
    b = P.Batch(None, 2, 16, max_draft_len=8, vocab=5)
    dev = b.device
    toks, cnt = _t([[1, 2], [3, 4]], dev), _t([2, 2], dev)
    out = P.StepOutputs(2, 8, dev)
    L = P.lib()
    args = [toks.data_ptr(), 2, cnt.data_ptr(), 8] + [t.data_ptr() for t in out.tensors()] + [None]
    assert L.sam_step(b.handle, *args) == 0
    bad = list(args); bad[3] = 9                                   # L > max_draft_len
    assert L.sam_step(b.handle, *bad) == -1
    bad = list(args); bad[1] = 0                                   # stride < 1
    assert L.sam_step(b.handle, *bad) == -1
    bad = list(args); bad[4] = None                                # null output
    assert L.sam_step(b.handle, *bad) == -1
    ws = torch.empty(1024, dtype=torch.uint8, device=dev)
    h = P.binding.c_void_p()
    o = P.BatchOpts(2, 16, 8, 0, 1, 5, 0, 0, 0)
    assert L.sam_batch_create(None, P.binding.byref(o), ws.data_ptr(), ws.numel(), None, P.binding.byref(h)) == -4
    torch.cuda.synchronize()
    assert batch_ok(P, b)


def batch_ok(P, b):
    tot, free = b.pool_info()
    return 0 <= free <= tot


def test_reset_returns_slabs_and_slots_restart(P):
    import torch
    rng = random.Random(3)
    vocab, n, L, B = 40, 600, 8, 6
    texts = [[rng.randrange(vocab) for _ in range(n)] for _ in range(B)]
    nt = np.array(texts, dtype=np.int32)
    b = P.Batch(None, B, n, max_draft_len=L, vocab=vocab, slab_bytes=4096)
    tot, free0 = b.pool_info()
    assert free0 == tot
    full = np.full(B, n, dtype=np.int32)
    o1 = b.step(_t(nt, b.device), _t(full, b.device), L).cpu()
    _, free1 = b.pool_info()
    assert free1 < free0
    b.reset([1, 4])
    _, free2 = b.pool_info()
    assert free1 < free2 < free0
    # slots 1 and 4 start over with other text; the rest are untouched (count 0 re-emits)
    nt2 = nt.copy(); nt2[1] = nt[2]; nt2[4] = nt[0]
    cnt = np.zeros(B, dtype=np.int32); cnt[[1, 4]] = n
    o2 = b.step(_t(nt2, b.device), _t(cnt, b.device), L).cpu()
    for k in KEYS:
        assert np.array_equal(o2[k][[0, 2, 3, 5]], o1[k][[0, 2, 3, 5]]), k
        assert np.array_equal(o2[k][1], o1[k][2]) and np.array_equal(o2[k][4], o1[k][0]), k
    b.reset()
    _, free3 = b.pool_info()
    assert free3 == tot
    o3 = b.step(_t(nt, b.device), _t(full, b.device), L).cpu()
    for k in KEYS:
        assert np.array_equal(o3[k], o1[k])


def test_pool_exhaustion_is_a_status_not_a_fault(P):
    rng = random.Random(4)
    vocab, n, L, B = 500, 2000, 8, 4
    nt = np.array([[rng.randrange(vocab) for _ in range(n)] for _ in range(B)], dtype=np.int32)
    b = P.Batch(None, B, n, max_draft_len=L, vocab=vocab, slab_bytes=4096, pool_slabs=20)
    o = b.step(_t(nt, b.device), _t(np.full(B, n), b.device), L).cpu()
    assert (o["status"] == 1).any()                     # 4 x 2000 tokens cannot fit 20 slabs of 4 KiB
    assert set(o["status"].tolist()) <= {0, 1}
    assert (o["draft_len"][o["status"] == 1] == 0).all()
    o2 = b.step(_t(nt[:, :1], b.device), _t(np.zeros(B), b.device), L).cpu()
    assert np.array_equal(o2["status"], o["status"])   # sticky
    b.reset()
    ok = b.step(_t(nt[:, :50], b.device), _t(np.full(B, 50), b.device), L).cpu()
    assert (ok["status"] == 0).all()


def test_host_step_equals_device_step(P):
    import torch
    spec = W.scaled(W.SPECS["tiny"], corpus_len=30000, batch=5, prompt_len=40, gen_len=120)
    w = W.make(spec)
    L, msl = spec.draft_len, spec.prompt_len + spec.gen_len
    st = P.StaticSam.build(w.corpus, spec.vocab)
    ref, _, _ = oracle_run(w.corpus, spec.vocab, w.prompts, w.new_tokens, w.counts, L, msl)
    b = P.Batch(st, spec.batch, msl, max_draft_len=L, max_host_stride=spec.prompt_len)
    B = spec.batch
    mk = lambda *s: torch.empty(s, dtype=torch.int32).pin_memory()
    out = dict(draft_tokens=mk(B, L), draft_len=mk(B), match_len=mk(B, 2), source=mk(B), state=mk(B, 2), status=mk(B))
    steps = [(w.prompts, np.full(B, spec.prompt_len, dtype=np.int32))] + \
            [(w.new_tokens[s], w.counts[s]) for s in range(w.n_steps)]
    prepared = {}                                       # the bound form of the call, one per stride
    for i, (toks, cnt) in enumerate(steps):
        toks = np.ascontiguousarray(toks)
        if i % 2 == 0:
            P.binding.sam_step_host(b.handle, toks, toks.shape[1], np.ascontiguousarray(cnt), L,
                                    *[out[k] for k in KEYS])
        else:
            if toks.shape[1] not in prepared:
                prepared[toks.shape[1]] = P.binding.sam_step_host_prepared(b.handle, toks.shape[1], L, *[out[k] for k in KEYS])
            prepared[toks.shape[1]](toks, np.ascontiguousarray(cnt))
        for k in KEYS:
            assert np.array_equal(out[k].numpy(), ref[k][i]), (i, k)
    with pytest.raises(P.SamError):
        big = np.zeros((B, spec.prompt_len + 1), dtype=np.int32)
        P.binding.sam_step_host(b.handle, big, big.shape[1], np.zeros(B, np.int32), L, *[out[k] for k in KEYS])


@pytest.mark.parametrize("B", [600, 1700, 8300])
def test_host_step_large_with_pinned_and_pageable_arrays(P, B):
    """Large host steps: page-locked caller arrays are read and written in place, pageable ones go
    through the staging area (and, at this size, two DMA copies or the mapped staging area — the DMA path
    runs the device step as it is: slot ordering at 1700 slots, the split step at 8300; the in-place paths
    run one unordered two-warp launch whatever the batch).  All equal the oracle."""
    import torch
    spec = W.scaled(W.SPECS["c5"], corpus_len=60_000, batch=B, prompt_len=24, gen_len=40)
    w = W.make(spec)
    L, msl = spec.draft_len, spec.prompt_len + spec.gen_len
    st = P.StaticSam.build(w.corpus, spec.vocab)
    ref, _, _ = oracle_run(w.corpus, spec.vocab, w.prompts, w.new_tokens, w.counts, L, msl, threads=4)
    steps = [(w.prompts, np.full(B, spec.prompt_len, dtype=np.int32))] + \
            [(w.new_tokens[s], w.counts[s]) for s in range(w.n_steps)]
    for pinned in (True, False):
        b = P.Batch(st, B, msl, max_draft_len=L, max_host_stride=spec.prompt_len)
        mk = (lambda *s: torch.empty(s, dtype=torch.int32).pin_memory()) if pinned else (lambda *s: torch.empty(s, dtype=torch.int32))
        out = dict(draft_tokens=mk(B, L), draft_len=mk(B), match_len=mk(B, 2), source=mk(B), state=mk(B, 2), status=mk(B))
        for i, (toks, cnt) in enumerate(steps):
            t = torch.from_numpy(np.ascontiguousarray(toks)); c = torch.from_numpy(np.ascontiguousarray(cnt))
            if pinned:
                t, c = t.pin_memory(), c.pin_memory()
            P.binding.sam_step_host(b.handle, t, t.shape[1], c, L, *[out[k] for k in KEYS])
            for k in KEYS:
                assert np.array_equal(out[k].numpy(), ref[k][i]), (pinned, i, k)
        b.close()


def test_cached_static_automaton_is_built_once_then_loaded(P, tmp_path):
    """StaticSam.cached keeps the built image under a name derived from the corpus: the first call builds and
    saves, the second loads the same automaton, another corpus gets another file, a damaged file is rebuilt."""
    spec = W.scaled(W.SPECS["c2"], corpus_len=90_000, batch=3, prompt_len=60, gen_len=120)
    w = W.make(spec)
    L, msl = spec.draft_len, spec.prompt_len + spec.gen_len
    d = str(tmp_path / "cache")
    st1, how1 = P.StaticSam.cached(w.corpus, spec.vocab, d)
    st2, how2 = P.StaticSam.cached(w.corpus, spec.vocab, d)
    assert (how1, how2) == ("built", "loaded") and len(os.listdir(d)) == 1
    r1, _ = gpu_run(P, st1, spec.vocab, w.prompts, w.new_tokens, w.counts, L, msl)
    r2, _ = gpu_run(P, st2, spec.vocab, w.prompts, w.new_tokens, w.counts, L, msl)
    assert_same(r2, r1)
    other = w.corpus.copy(); other[5] = (other[5] + 1) % spec.vocab
    _, how3 = P.StaticSam.cached(other, spec.vocab, d)
    assert how3 == "built" and len(os.listdir(d)) == 2
    path = os.path.join(d, sorted(os.listdir(d))[0])
    raw = bytearray(open(path, "rb").read()); raw[len(raw) // 2] ^= 0x10
    open(path, "wb").write(bytes(raw))
    hows = {P.StaticSam.cached(c, spec.vocab, d)[1] for c in (w.corpus, other)}
    assert hows == {"built", "loaded"}                      # the damaged one was rebuilt, the other loaded


def test_image_save_load_roundtrip(P, tmp_path):
    spec = W.scaled(W.SPECS["c2"], corpus_len=120_000, batch=4, prompt_len=100, gen_len=200)
    w = W.make(spec)
    L, msl = spec.draft_len, spec.prompt_len + spec.gen_len
    st = P.StaticSam.build(w.corpus, spec.vocab)
    path = str(tmp_path / "static.sam")
    st.save(path)
    st2 = P.StaticSam.load(path)
    a, b = st.info, st2.info
    assert (a.n_states, a.n_transitions, a.hash_buckets, a.vocab) == (b.n_states, b.n_transitions, b.hash_buckets, b.vocab)
    r1, _ = gpu_run(P, st, spec.vocab, w.prompts, w.new_tokens, w.counts, L, msl)
    r2, _ = gpu_run(P, st2, spec.vocab, w.prompts, w.new_tokens, w.counts, L, msl)
    assert_same(r2, r1)
    raw = bytearray(open(path, "rb").read())
    raw[len(raw) // 2] ^= 0x40
    open(path, "wb").write(bytes(raw))
    with pytest.raises(P.SamError) as e:
        P.StaticSam.load(path)
    assert e.value.code == -6
    with pytest.raises(P.SamError) as e:
        P.StaticSam.load(str(tmp_path / "missing.sam"))
    assert e.value.code == -5


def test_static_tables_match_oracle_on_device(P):
    spec = W.scaled(W.SPECS["tiny"], corpus_len=50_000)
    corpus = W.make_corpus(spec)
    st = P.StaticSam.build(corpus, spec.vocab)
    S = oracle.Sam(corpus)
    link, length, endpos, deg = S.tables()
    tb = P.binding.sam_static_tables(st.handle)
    assert np.array_equal(tb["length"], length) and np.array_equal(tb["link"], link)
    assert np.array_equal(tb["min_endpos"], endpos) and np.array_equal(tb["deg"], deg)
    busiest = np.argsort(deg)[-5:].tolist()
    rng = random.Random(0)
    for s in busiest + [rng.randrange(S.n_states) for _ in range(30)]:
        got = P.binding.sam_static_state(st.handle, s, max_edges=int(deg[s]) + 1)
        assert got["next"] == S.edges(s), s


def test_probes_report_plausible_numbers(P):
    import torch
    buf = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for g in (32, 64, 128):
        gbps, mreq = P.binding.sam_probe_random_read(buf, g, iters=2)
        assert 10 < gbps < 20000 and mreq > 0
    ns1 = P.binding.sam_probe_chase(buf, 20000, chains=1)
    ns64 = P.binding.sam_probe_chase(buf, 20000, chains=64)
    assert 100 < ns1 < 5000 and 100 < ns64 < 5000


def test_stop_token_matches_oracle(P):
    spec = W.scaled(W.SPECS["tiny"], corpus_len=40_000, batch=6, prompt_len=100, gen_len=300)
    w = W.make(spec)
    L, msl = 40, spec.prompt_len + spec.gen_len
    vals, cnts = np.unique(w.corpus, return_counts=True)
    stop = int(vals[np.argmax(cnts)])                       # the most frequent token plays the separator
    st = P.StaticSam.build(w.corpus, spec.vocab)
    ref, _, _ = oracle_run(w.corpus, spec.vocab, w.prompts, w.new_tokens, w.counts, L, msl, stop_token=stop)
    got, _ = gpu_run(P, st, spec.vocab, w.prompts, w.new_tokens, w.counts, L, msl, stop_token=stop)
    assert_same(got, ref)
    plain, _ = gpu_run(P, st, spec.vocab, w.prompts, w.new_tokens, w.counts, L, msl)
    assert (got["draft_len"] < plain["draft_len"]).any()    # some drafts were cut
    assert not (got["draft_tokens"] == stop).any()


def test_per_step_calls_without_the_extension_module(P, monkeypatch):
    """A machine that cannot compile csrc/calls.c: every call it marshals gives the same results through ctypes."""
    import torch
    rng = np.random.default_rng(12)
    vocab, B, n, L = 30, 6, 80, 8
    corpus = rng.integers(0, vocab, size=3000, dtype=np.int32)
    st = P.StaticSam.build(corpus, vocab, tree_topk=3)
    toks = torch.from_numpy(rng.integers(0, vocab, size=(B, n), dtype=np.int32)).cuda()
    counts, few = (torch.full((B,), k, dtype=torch.int32, device="cuda") for k in (n, 5))
    x = P.binding

    def all_calls():
        i32 = dict(dtype=torch.int32, device="cuda")
        b = P.Batch(st, B, 4 * n, max_draft_len=L)
        first, second, host = b.step(toks, counts, L), P.StepOutputs(B, L, "cuda"), P.StepOutputs(B, L, "cpu")
        x.sam_step(b.handle, toks[:, :5].contiguous(), 5, few, L, *second.tensors())
        new, cnt, acc = torch.empty(B, L + 1, **i32), torch.empty(B, **i32), torch.empty(B, **i32)
        target = torch.cat([first.draft_tokens, first.draft_tokens[:, :1]], 1).clamp_(0, vocab - 1).contiguous()
        x.sam_accept_greedy(first.draft_tokens, first.draft_len, target, None, new, cnt, acc)
        third = P.StepOutputs(B, L, "cuda")
        x.sam_step_verified(b.handle, target, first.draft_tokens, first.draft_len, None, L, *third.tensors(), counts_out=cnt, accepted_out=acc)
        x.sam_select_auxiliary(third.draft_tokens, third.draft_len, third.source, target[:, :L].contiguous(), few)
        x.sam_step_host(b.handle, toks[:, :5].cpu(), 5, few.cpu(), L, *host.tensors())
        again = P.StepOutputs(B, L, "cpu")
        x.sam_step_host_prepared(b.handle, 5, L, *again.tensors())(toks[:, 5:10].cpu().contiguous(), few.cpu())
        tree = [torch.empty(B, 12, **i32), torch.empty(B, 12, **i32), torch.empty(B, 12, device="cuda"), torch.empty(B, **i32)]
        x.sam_tree_draft(st.handle, first.state[:, 0].contiguous(), toks[:, -1].contiguous(), 12, 3, *tree)
        once = P.StepOutputs(B, L, "cuda")
        x.sam_retrieve_noalloc(st.handle, vocab, toks, counts, L, 0, 1, *once.tensors())
        return [t.cpu().numpy() for o in (first, second, third, host, again, once) for t in o.tensors()] + [t.cpu().numpy() for t in (new, cnt, acc, *tree)]

    expected = all_calls()

    def build_calls(force=False):
        raise FileNotFoundError("gcc")

    monkeypatch.setattr(x, "_calls", None)
    monkeypatch.setattr(x, "_fn", {})
    monkeypatch.setattr(x._build, "build_calls", build_calls)
    with pytest.warns(RuntimeWarning, match="ctypes"):
        got = all_calls()
    assert x._calls is x._PlainCalls
    assert len(got) == len(expected) and all(np.array_equal(a, b) for a, b in zip(got, expected))


@pytest.mark.parametrize("B,K,L", [(100, 40, 128), (200, 16, 128), (700, 8, 24)])
def test_host_arrays_are_the_callers_again_when_the_call_returns(P, B, K, L):
    """Page-locked arrays that kernels work on in place (64 KiB and more in all, rows too few to be fetched ahead): every step has
    arrays of its own, unregistered and overwritten as soon as the call returns; the batch is dropped after the last."""
    import torch
    assert B * (K + 1) < 8192 and B * (K + 1 + L + 7) * 4 >= 65536
    rt = torch.cuda.cudart()
    rng = np.random.default_rng(B)
    vocab, steps = 30, 12
    corpus = rng.integers(0, vocab, size=4000, dtype=np.int32)
    st, S = P.StaticSam.build(corpus, vocab), oracle.Sam(corpus)
    ob, batch = oracle.Batch(S, corpus, B, vocab, K * steps), P.Batch(st, B, K * steps, max_draft_len=L, max_host_stride=K)
    shapes = ((B, K), (B,), (B, L), (B,), (B, 2), (B,), (B, 2), (B,))
    words = [int(np.prod(s)) for s in shapes]
    for i in range(steps):
        toks = rng.integers(0, vocab, size=(B, K), dtype=np.int32)
        counts = rng.integers(0, K + 1, size=B).astype(np.int32)
        raw = np.full(sum(words) + 1024, -9, dtype=np.int32)
        at = (-(raw.ctypes.data // 4)) % 1024                # a page of its own
        assert int(rt.cudaHostRegister(raw.ctypes.data + 4 * at, 4 * sum(words), 0)) == 0
        views = []
        for s, n in zip(shapes, words):
            views.append(raw[at:at + n].reshape(s)); at += n
        views[0][:], views[1][:] = toks, counts
        P.binding.sam_step_host(batch.handle, views[0], K, views[1], L, *views[2:])
        assert int(rt.cudaHostUnregister(views[0].ctypes.data)) == 0
        got = [v.copy() for v in views[2:]]
        raw[:] = -5
        ref = ob.step(toks, counts, L, 4)
        for k, v in zip(KEYS, got):
            assert np.array_equal(v, getattr(ref, k)), (i, k)
    batch.close()


@pytest.mark.parametrize("B,K,L", [(1, 8, 16), (16, 60, 16), (60, 16, 32), (64, 100, 50), (300, 12, 40), (1300, 8, 24)])
def test_a_host_step_is_followed_by_work_on_another_stream(P, B, K, L):
    """Nothing but the host call's return orders the stream of the next call behind it: device steps, dumps and resets there see
    the batch as the host step left it, prompts (rows of 60 and 100) included."""
    import torch
    rng = np.random.default_rng(B)
    vocab, rounds, msl = 12, 25, 400
    corpus = rng.integers(0, vocab, size=4000, dtype=np.int32)
    st, S = P.StaticSam.build(corpus, vocab), oracle.Sam(corpus)
    batch = P.Batch(st, B, msl, max_draft_len=L, max_host_stride=K)
    streams = [torch.cuda.Stream() for _ in range(2)]
    ob = oracle.Batch(S, corpus, B, vocab, msl)
    out = [np.empty(s, dtype=np.int32) for s in ((B, L), (B,), (B, 2), (B,), (B, 2), (B,))]
    dev = P.StepOutputs(B, L, "cuda")
    torch.cuda.synchronize()
    for i in range(rounds):
        toks = rng.integers(0, vocab, size=(2, B, K), dtype=np.int32)
        counts = np.stack([np.full(B, K if i % 3 == 0 else 3), rng.integers(0, 3, size=B)]).astype(np.int32)
        d = [torch.from_numpy(x).cuda() for x in (toks[1], counts[1])]
        torch.cuda.synchronize()
        P.binding.sam_step_host(batch.handle, toks[0], K, counts[0], L, *out, stream=streams[0])
        with torch.cuda.stream(streams[1]):
            P.binding.sam_step(batch.handle, d[0], K, d[1], L, *dev.tensors(), stream=streams[1])
            ref = ob.step(toks[0], counts[0], L, 4)
            for k, v in zip(KEYS, out):
                assert np.array_equal(v, getattr(ref, k)), (i, k)
            ref = ob.step(toks[1], counts[1], L, 4)
            streams[1].synchronize()
        for k, v in dev.cpu().items():
            assert np.array_equal(v, getattr(ref, k)), (i, k)
        if i % 3 == 2:                                      # start over: the next host step brings prompts again
            P.binding.sam_batch_reset(batch.handle, None, streams[0])
            streams[0].synchronize()
            ob = oracle.Batch(S, corpus, B, vocab, msl)
