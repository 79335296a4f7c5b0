"""After a route that failed between its kernels, the next calls start from an
empty group table: routes and session links as if the failed one had not been."""

import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2607_08565_gb300 as pkg
from gpu_util import T, assert_outputs_equal, gpu_route, make_index, populate_both
from synth.traces import pack

pytestmark = pytest.mark.gpu
MASK_WORDS_AT = ctypes.sizeof(pkg.smetric_index_config) + 8  # in the index: its configuration, the device, its SMs, then W


def test_calls_after_a_route_that_failed_halfway():
    rng = np.random.default_rng(5)
    N, B, n = 3, 2, 32
    ix = make_index(N, B, 2, max_req=n, max_tok=40 * n)
    ox = oracle.OracleIndex(N)
    pool = rng.integers(0, 99, size=30, dtype=np.int32)
    populate_both(ix, ox, {-1: [pool], 1: [pool[:20]]}, B)
    load = np.zeros(N, np.int64)
    # no host code takes 9 mask words: the call returns after the digest has filled the group table
    words = ctypes.c_int.from_address(ix.handle + MASK_WORDS_AT)
    assert words.value == 1
    for k in range(2):  # 64 first blocks: as many as the table has places
        tok = np.arange(n * B, dtype=np.int32) + 1000 * (k + 1)
        words.value = 9
        with pytest.raises(pkg.SmetricError):
            ix.route_batch(T(tok), T(np.arange(n + 1, dtype=np.int64) * B), T(load), (1, 4, 2))
        words.value = 1
    users, turns = np.arange(n, dtype=np.int64) % 8, (np.arange(n) // 8).astype(np.int32)
    reqs = [pool[:4 + 6 * t + u % 3 * 2] for u, t in zip(users, turns)]
    tok, off = pack(reqs)
    parent, session = ix.link_sessions(T(tok), T(off), T(users), T(turns))
    ix.check()
    want = oracle.link_sessions(B, 0, tok, off, users, turns)
    assert np.array_equal(parent.cpu().numpy(), want[0]) and np.array_equal(session.cpu().numpy(), want[1])
    assert (want[0] >= 0).any()
    assert_outputs_equal(gpu_route(ix, tok, off, load, (1, 4, 2)), ox.route_batch(B, 2, 0, tok, off, load, 1, 4, 2, want_hashes=True))
    ix.close()
