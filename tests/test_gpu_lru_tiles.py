"""The device LRU at the edges of its tiles (1,024 records or touches) and of its
plan's rounds (1,024 requests), against the LRU oracle: after every commit
every key seen is in exactly the tiers that the oracle keeps it in."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from gpu_util import T, make_index

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,local_cap,global_cap", [(5, 1023, 0), (5, 1024, 1025), (70, 40, 2047), (256, 0, 1024)])
def test_lru_tiles_and_plan_rounds(N, local_cap, global_cap):
    rng = np.random.default_rng(N + local_cap)
    B = 2
    ix = make_index(N, B, 1, cap=1 << 16, max_req=2100, max_tok=2100 * 5 * B)
    ix.set_lru(local_cap, global_cap)
    ol = oracle.OracleLRU(N, local_cap=local_cap, global_cap=global_cap)
    pool = np.unique(rng.integers(2, 1 << 63, size=9000, dtype=np.uint64))
    rng.shuffle(pool)
    seen = set()
    for step, n in enumerate((1, 1023, 1024, 1025, 2100, 1100, 300)):
        nblk = rng.integers(0, 5, size=n)
        off = np.zeros(n + 1, np.int64)
        np.cumsum(nblk * B, out=off[1:])
        # a herd to one instance, or spread over all; keys come again within and across batches
        inst = (np.full(n, step % N) if step % 2 else rng.integers(-1, N, size=n)).astype(np.int32)
        lo = int(rng.integers(0, 4000))
        h = pool[rng.integers(lo, lo + 4500, size=int(nblk.sum()))]
        out = dict(instance=T(inst), local_hit=T(np.zeros(n, np.int32)), block_hashes=T(np.append(h, np.uint64(2))))
        ix.commit_batch(T(off), out, also_global=True)
        ix.check()
        on = inst >= 0
        held = np.concatenate([np.full(k, b) for k, b in zip(nblk, on)]).astype(bool) if n else np.zeros(0, bool)
        ol.commit(nblk[on], inst[on], h[held], also_global=True)
        seen.update(h[held].tolist())
        sizes = ix.lru_sizes().cpu().numpy().tolist()
        assert sizes == [ol.size(i) for i in range(N)] + [ol.size(-1)]
        keys = np.array(sorted(seen), np.uint64)
        m = ix.lookup(T(keys)).cpu().numpy().view(np.uint64)
        for t in ([*range(N)] if local_cap else []) + ([-1] if global_cap else []):
            bit = N if t < 0 else t
            got = keys[(m[:, bit >> 6] >> np.uint64(bit & 63)) & np.uint64(1) == 1]
            assert set(got.tolist()) == set(ol.stamp[t]), (step, t)
    ix.close()
