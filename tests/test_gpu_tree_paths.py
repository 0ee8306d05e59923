"""GPU: trees that run along passages the corpus holds several times — paths shorter and longer than a round of 32 and than
the largest tree, ending in a choice, in a state with many successors and at the corpus' end — against the oracle."""
import random

import numpy as np
import pytest

import oracle
from test_gpu_tree import P, _check  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length", [1, 2, 31, 32, 33, 127, 128, 300])
def test_paths_of_every_length(P, length, tmp_path):  # noqa: F811
    rng = random.Random(length)
    vocab = 5000
    x = []
    for _ in range(4):                                       # four passages, each three to five times, with different tokens after
        passage = [rng.randrange(vocab) for _ in range(length)]
        for _ in range(rng.randint(3, 5)):
            x += [rng.randrange(3)] + passage + [rng.randrange(vocab)]
    passage = [rng.randrange(vocab) for _ in range(length)]
    for t in list(range(40)) + [None]:                       # one with many successors, the last of them none
        x += passage + ([t] if t is not None else [])
    x = np.array(x, dtype=np.int32)
    S = oracle.Sam(x)
    f = S.freq()
    built = P.StaticSam.build(x, vocab, tree_topk=4)
    built.save(str(tmp_path / "image"))
    states = [0, 1, S.n_states - 1] + [rng.randrange(1, S.n_states) for _ in range(60)]
    starts = [rng.randrange(vocab) for _ in states]
    for st in (built, P.StaticSam.load(str(tmp_path / "image"))):
        for max_size, k in ((128, 4), (40, 2), (33, 1), (5, 4)):
            _check(P, S, f, st, states, starts, max_size, k)


@pytest.mark.parametrize("fan", [(1, 1), (2, 3), (5, 6), (6, 6)])
@pytest.mark.parametrize("repeats", [1, 2, 3])
def test_many_equally_probable_entries(P, fan, repeats):  # noqa: F811
    """Up to 36 entries of one probability in the queue: paths of several lengths, states with a choice after one token, and
    both in one line, in the order in which they were pushed."""
    rng = random.Random(fan[0] * 10 + fan[1] + repeats)
    x, s = [], 5000
    for i in range(fan[0]):
        for j in range(fan[1]):
            tail = [rng.randrange(100, 5000) for _ in range((i + j) % 5)]
            for _ in range(repeats):
                x += [s, 10 + i, 30 + j] + tail + [rng.randrange(100, 5000), 6000 + len(x) % 900]
    x = np.array(x, dtype=np.int32)
    S = oracle.Sam(x)
    st = P.StaticSam.build(x, 8000, tree_topk=6)
    states = [S.edges(0)[s]] * 2 + [rng.randrange(1, S.n_states) for _ in range(30)]
    starts = [rng.randrange(8000) for _ in states]
    for max_size, k in ((128, 6), (50, 5), (9, 6), (2, 1)):
        _check(P, S, S.freq(), st, states, starts, max_size, k)
