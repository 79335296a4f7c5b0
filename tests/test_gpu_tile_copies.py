"""Block digests through the tile copies: requests at every token phase, chunks
that end with the buffer or a block before it, buffers too short for a tile,
against the oracle."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from gpu_util import T, gpu_hashes, make_index
from synth.traces import pack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [16, 32, 64, 128])
def test_digests_at_every_phase_and_buffer_end(B):
    rng = np.random.default_rng(B)
    ix = make_index(3, B, 2, max_tok=70 * B + 200)
    for shift in [*range(0, B, 4), 1, 2, 3, B - 1, B + 1]:
        # blocks of the last request, and the tokens of the buffer after it
        for blocks, rest in ((1, 0), (1, B - shift % B), (2, 1), (31, 4), (32, 0), (32, B), (33, B - 4), (66, 2 * B)):
            tok = rng.integers(0, 151936, size=shift + blocks * B + rest, dtype=np.int32)
            off = np.array([0, shift, shift + blocks * B], np.int64)
            hb, sk = gpu_hashes(ix, tok, off)
            h = [oracle.block_hashes(tok[a:b], B) for a, b in zip(off[:-1], off[1:])]
            assert np.array_equal(hb, np.concatenate(h)), (shift, blocks, rest)
            assert np.array_equal(sk, np.array([x[min(len(x), 2) - 1] if len(x) else 0 for x in h], np.uint64))
    ix.close()
