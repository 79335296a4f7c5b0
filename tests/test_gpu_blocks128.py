"""Blocks of 128 tokens through the tile copies: ragged requests at every token
phase, chunks that end with the buffer, short and long requests, against the
oracle."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from gpu_util import assert_outputs_equal, gpu_hashes, gpu_route, make_index, populate_both
from synth.traces import pack

pytestmark = pytest.mark.gpu
B = 128


@pytest.mark.parametrize("lens", [
    [1, 2, 3, 127, 128, 129, 255, 256, 4095, 4096, 4097, 31 * 128, 33 * 128 + 1],
    [5, 32 * 128], [7, 32 * 128 + 64], [0, 128], [3 * 128 - 1], [9, 70 * 128 + 3, 1, 32 * 128],
])
def test_digests_at_every_phase_and_the_buffer_end(lens):
    rng = np.random.default_rng(sum(lens))
    for shift in range(5):
        reqs = [rng.integers(0, 151936, size=shift, dtype=np.int32)] + \
               [rng.integers(0, 151936, size=n, dtype=np.int32) for n in lens]
        tok, off = pack(reqs)
        ix = make_index(3, B, 2, max_tok=max(len(tok), 1))
        hb, sk = gpu_hashes(ix, tok, off)
        h = [oracle.block_hashes(r, B) for r in reqs]
        assert np.array_equal(hb, np.concatenate(h))
        assert np.array_equal(sk, np.array([x[min(len(x), 2) - 1] if len(x) else 0 for x in h], np.uint64))
        ix.close()


def test_route_of_many_and_long_requests():
    rng = np.random.default_rng(7)
    N = 9
    base = rng.integers(0, 151936, size=90 * B, dtype=np.int32)
    reqs = [np.concatenate([base[:int(rng.integers(0, 90 * B))], rng.integers(0, 9, size=int(rng.integers(0, 900)),
                                                                              dtype=np.int32)]) for _ in range(900)]
    reqs += [rng.integers(0, 151936, size=200000, dtype=np.int32)]
    tok, off = pack(reqs)
    ix = make_index(N, B, 2, max_tok=len(tok))
    ox = oracle.OracleIndex(N)
    populate_both(ix, ox, {-1: [base], 2: [base[:40 * B], reqs[-1]], 8: [base[:41 * B]]}, B)
    load = rng.integers(0, 9000, size=N)
    g = gpu_route(ix, tok, off, load, (1, 4, 2))
    o = ox.route_batch(B, 2, 0, tok, off, load, 1, 4, 2, want_hashes=True)
    assert_outputs_equal(g, o)
    ix.close()
