"""The reuse breakdown between its samples: prompts of 1 to 1,100 blocks (the
samples are every block up to 32, and more than 32 blocks apart past 1,024)
that share prefixes of any length across sessions, against the oracle."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from gpu_util import T, make_index
from synth.traces import pack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("longest", [1, 31, 32, 33, 65, 1023, 1024, 1025, 1100])
def test_holders_change_anywhere(longest):
    rng = np.random.default_rng(longest)
    B, n = 2, 90
    texts = [rng.integers(0, 150000, size=B * longest, dtype=np.int32) for _ in range(2)]
    reqs, sessions = [], []
    for r in range(n):
        t = texts[int(rng.integers(2))]
        k = int(rng.integers(0, longest + 1)) if r % 3 else longest
        own = rng.integers(0, 150000, size=B * int(rng.integers(0, max(1, longest - k + 1))) + int(rng.integers(0, 2)),
                           dtype=np.int32)
        reqs.append(np.concatenate([t[:B * k], own]))
        sessions.append(int(rng.integers(0, 6)))
    tok, off = pack(reqs)
    sys_blocks = rng.integers(0, longest + 2, size=n).astype(np.int32)
    sess = np.array(sessions, np.int32)
    ix = make_index(2, B, 1, max_req=n, max_tok=len(tok) + 8)
    out = ix.reuse_breakdown(T(tok), T(off), T(sess), T(sys_blocks))
    ix.check()
    o = oracle.reuse_breakdown(B, 0, tok, off, sess, sys_blocks)
    for k in ("hit", "sys", "intra", "inter"):
        assert np.array_equal(out[k].cpu().numpy(), o[k]), k
    ix.close()
