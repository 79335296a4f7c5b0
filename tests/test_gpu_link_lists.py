"""Session links where their search changes: turns with 64 and 65 requests (the
longest list that is gone through, and one more), chains of parents on both
sides of 64, against the oracle."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from gpu_util import T, make_index
from synth.traces import pack

pytestmark = pytest.mark.gpu


def _check(ix, reqs, users, turns, B):
    tok, off = pack(reqs)
    parent, session = ix.link_sessions(T(tok), T(off), T(np.asarray(users, np.int64)), T(np.asarray(turns, np.int32)))
    ix.check()
    op, os_ = oracle.link_sessions(B, 0, tok, off, np.asarray(users, np.int64), np.asarray(turns, np.int32))
    assert np.array_equal(parent.cpu().numpy(), op)
    assert np.array_equal(session.cpu().numpy(), os_)
    return op


@pytest.mark.parametrize("size", [1, 63, 64, 65, 300])
def test_lists_of_a_turn(size):
    rng = np.random.default_rng(size)
    B = 2
    base = rng.integers(0, 5, size=60, dtype=np.int32)
    reqs, users, turns = [], [], []
    for user, count in ((1, size), (2, 3), (-7, size)):
        for turn in (0, 1, 2):
            for _ in range(count if turn < 2 else 5):
                n = int(rng.integers(0, 50))
                reqs.append(np.concatenate([base[:n], rng.integers(0, 5, size=int(rng.integers(0, 6)), dtype=np.int32)]))
                users.append(user)
                turns.append(turn)
    order = rng.permutation(len(reqs))
    ix = make_index(2, B, 1, max_req=len(reqs), max_tok=len(reqs) * 60)
    for o in (np.arange(len(reqs)), order):
        op = _check(ix, [reqs[i] for i in o], [users[i] for i in o], [turns[i] for i in o], B)
    assert size < 63 or (op >= 0).any()
    ix.close()


@pytest.mark.parametrize("depth", [2, 63, 64, 65, 66, 130, 700])
def test_long_chains_of_turns(depth):
    rng = np.random.default_rng(depth)
    B = 2
    text = rng.integers(0, 9, size=2 * depth + 4, dtype=np.int32)
    reqs = [text[:2 * t + 2] for t in range(depth)] + [rng.integers(0, 9, size=5, dtype=np.int32)]
    ix = make_index(2, B, 1, max_req=len(reqs), max_tok=sum(map(len, reqs)) + 8)
    op = _check(ix, reqs, [3] * depth + [4], list(range(depth)) + [1], B)
    assert np.array_equal(op[:depth], np.arange(-1, depth - 1))
    ix.close()
