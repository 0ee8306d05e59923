"""CPU model of the static side of replayed steps (csrc/step.cu, static_chunk) against the longest suffix by definition.

All suffixes that begin in a chunk of tokens are walked side by side, one lane each, and one lane is the match so far; what holds
after a token is what the lanes leave in one shared array, in an order that the scheme has to get right.  The model runs the
scheme a round at a time over dictionaries.  Stores of one round that no barrier separates take effect in any order,
so where the result depended on it some order gives a wrong one.
"""
import random

import pytest

LIMIT = 32


class Corpus:
    """Suffix automaton (Algorithm 3) with first end positions and the states of the prefixes."""

    def __init__(self, text):
        self.text, self.len, self.link, self.end, self.next, self.prefix = text, [0], [-1], [0], [{}], []
        last = 0
        for n, t in enumerate(text, 1):
            c = self._new(n, 0, n, {})
            p = last
            while p != -1 and t not in self.next[p]:
                self.next[p][t] = c
                p = self.link[p]
            if p != -1:
                q = self.next[p][t]
                if self.len[p] + 1 != self.len[q]:
                    k = self._new(self.len[p] + 1, self.link[q], self.end[q], dict(self.next[q]))
                    while p != -1 and self.next[p].get(t) == q:
                        self.next[p][t] = k
                        p = self.link[p]
                    self.link[q], q = k, k
                self.link[c] = q
            last = c
            self.prefix.append(c)

    def _new(self, ln, link, end, nx):
        self.len.append(ln); self.link.append(link); self.end.append(end); self.next.append(nx)
        return len(self.len) - 1


def follow(C, s, toks):
    """The run of transitions from state s that one round takes: [(state, first end position)], one for each token taken."""
    out = []
    if C.len[s] == C.end[s]:
        e = C.end[s]
        for k, t in enumerate(toks):
            if e + k >= len(C.text) or C.text[e + k] != t:
                break
            out.append((C.prefix[e + k], e + k + 1))
    elif toks and toks[0] in C.next[s]:
        d = C.next[s][toks[0]] - s
        at = s
        for t in toks if d in (1, 2) else []:
            if C.next[at].get(t) != at + d or len(C.next[at]) > 2:
                break
            at += d
            out.append((at, C.end[at]))
    return out


class Lane:
    def __init__(self, k):
        self.k, self.alive, self.have, self.need_len, self.came, self.chain = k, False, False, False, True, False
        self.s = self.l = 0
        self.pos = k + 1


def chunk(C, toks, ends, match, rng, barrier=True, guard=None):
    """One chunk: (match after it, results by token, tokens whose results hold, whether the links went on for too long)."""
    n, res = len(toks), {k: (0, 0, 0) for k in ends}
    lanes = [Lane(k) for k in range(32)]
    base = sure = 0
    for x in lanes[:n]:
        if toks[x.k] in C.next[0]:
            x.alive, x.s, x.l = True, C.next[0][toks[x.k]], 1
    if match[0]:
        x = lanes[0]
        x.chain = x.alive = x.have = True
        (x.s, x.l), x.pos = match, 0
    root = C.next[0].get(toks[0])
    guard = match[1] + 2 * n + 4 if guard is None else guard
    held, failed = n, False
    while True:
        live = [x for x in lanes if x.alive]
        arrived = next((x for x in live if x.pos == n), None)
        for x in live:
            if arrived and x.k > arrived.k:
                x.alive = False
        go = {x.k: x.alive and (x.pos < n or not x.have) for x in lanes}
        if not any(go.values()):
            break
        stores = []                                          # of this round, up to the next barrier
        fresh = {x.k: go[x.k] and not x.have for x in lanes}
        for x in lanes:
            if go[x.k]:
                x.have = True
                if x.need_len:
                    x.l, x.need_len = C.len[x.s], False
                if x.chain and x.pos - x.l >= max(base, 1):
                    x.alive = False
            go[x.k] = go[x.k] and x.alive and x.pos < n
            if fresh[x.k] and x.alive and x.came and x.pos > 0 and x.pos - 1 in ends and (x.chain or x.pos > sure):
                stores.append((x.pos - 1, (x.s, x.l, C.end[x.s])))
        tgt = {x.k: C.next[x.s].get(toks[x.pos]) if go[x.k] else None for x in lanes}
        first = next((x for x in lanes if x.alive), None)

        def settle():
            rng.shuffle(stores)
            for k, v in stores:
                res[k] = v
            stores.clear()

        if first is not None and go[first.k] and (first.chain or first.l >= 3):
            run, p0 = follow(C, first.s, toks[first.pos:]), first.pos
            if run:
                if barrier:
                    settle()
                stores += [(p0 + i, (s, first.l + i + 1, e)) for i, (s, e) in enumerate(run) if p0 + i in ends]
                base = sure = p0 + len(run)
                first.chain = first.came = True
                first.s, first.l, first.pos, first.have = run[-1][0], first.l + len(run), base, False
                go[first.k] = False
                for x in lanes[:base]:
                    if x is not first:
                        x.alive = go[x.k] = False
        for x in lanes:
            if not go[x.k]:
                continue
            x.have = x.came = False
            if tgt[x.k] is not None:
                x.s, x.l, x.pos, x.came = tgt[x.k], x.l + 1, x.pos + 1, True
            elif not x.chain:
                x.alive = False
            else:
                x.s = C.link[x.s]
                if x.s != 0:
                    x.need_len = True
                elif x.pos == 0 and root is not None:
                    x.s, x.l, x.pos, x.came = root, 1, 1, True
                else:
                    x.alive = False
                guard -= 1
                if guard < 0:
                    held, failed, x.alive = x.pos, True, False
        ahead = next((x for x in lanes if x.alive and x.chain), None)
        if ahead:
            sure = max(sure, 0 if ahead.need_len else ahead.pos)
        settle()
    x = next((x for x in lanes if x.alive), None)
    return ((x.s, x.l) if x else (0, 0)), res, held, failed


def longest(C, text):
    """(length, first end position) of the longest suffix of the text that occurs in the corpus, a token at a time (Algorithm 1)."""
    s = l = 0
    out = []
    for t in text:
        while s != 0 and t not in C.next[s]:
            s = C.link[s]
            l = C.len[s]
        if t in C.next[s]:
            s, l = C.next[s][t], l + 1
        out.append((s, l, C.end[s] if l else 0))
    return out


def texts(rng):
    """A corpus with passages that repeat, and a text that follows it in stretches of all lengths."""
    vocab = rng.choice([2, 3, 8, 60])
    corpus = [rng.randrange(vocab) for _ in range(rng.randint(20, 150))]
    for _ in range(rng.randint(0, 4)):
        a = rng.randrange(len(corpus))
        corpus += corpus[a:a + rng.randint(3, 50)]
    text = []
    while len(text) < 160:
        if rng.random() < 0.7:
            a = rng.randrange(len(corpus))
            text += corpus[a:a + rng.randint(1, 60)]
        else:
            text += [rng.randrange(vocab + 1) for _ in range(rng.randint(1, 6))]
    return corpus, text


def chunks_of(text, rng):
    at = 0
    while at < len(text):
        n = min(rng.randint(1, LIMIT), len(text) - at)
        yield at, text[at:at + n], {k for k in range(n) if k == n - 1 or rng.random() < 0.4}
        at += n


def wrong(seed, barrier):
    rng = random.Random(seed)
    corpus, text = texts(rng)
    C = Corpus(corpus)
    exp, match = longest(C, text), (0, 0)
    for at, toks, ends in chunks_of(text, rng):
        match, res, held, failed = chunk(C, toks, ends, match, rng, barrier)
        assert held == len(toks) and not failed
        if any(res[k] != exp[at + k] for k in ends) or match != exp[at + len(toks) - 1][:2]:
            return True
    return False


@pytest.mark.parametrize("seed", range(0, 400, 50))
def test_results_do_not_depend_on_the_order_of_stores(seed):
    assert not any(wrong(s, True) for s in range(seed, seed + 50))


def test_a_walk_ahead_and_the_run_that_overtakes_it_need_the_barrier():
    assert any(wrong(s, False) for s in range(400))


def test_what_holds_when_the_links_go_on_for_too_long():
    """A state whose link leads to itself: the results of the tokens before the one that it fails at hold."""
    seen = 0
    for seed in range(600):
        rng = random.Random(seed)
        corpus, text = texts(rng)
        C = Corpus(corpus)
        exp, match = longest(C, text), (0, 0)
        bad = rng.choice([s for s in range(1, len(C.len)) if C.len[s] > 2])
        C.link[bad] = bad
        for at, toks, ends in chunks_of(text, rng):
            match, res, held, failed = chunk(C, toks, ends, match, rng)
            for k in ends:
                assert k >= held or res[k] == exp[at + k], (seed, at, k)
            if failed:
                seen += held > min(ends)
                break
    assert seen > 20
