"""Refused block hashes (0 and 1) in commits on capped tiers: INVALID_ARG is
latched, the batch's other blocks are committed, and every tier keeps what the
LRU oracle keeps of those - on a first commit, after larger valid ones, and
after the tiers have been capped anew."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2607_08565_gb300 as pkg
from gpu_util import T, make_index

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,local_cap,global_cap", [(3, 40, 0), (3, 0, 100), (5, 1024, 700)])
def test_refused_hashes_take_no_place(N, local_cap, global_cap):
    rng = np.random.default_rng(N + local_cap)
    B, cap_req = 2, 900
    ix = make_index(N, B, 1, cap=1 << 15, max_req=cap_req, max_tok=cap_req * 6 * B)
    pool = np.unique(rng.integers(2, 1 << 63, size=4000, dtype=np.uint64))
    rng.shuffle(pool)
    seen = set()
    for caps in range(2):
        ix.clear()
        ix.set_lru(local_cap, global_cap)
        ol = oracle.OracleLRU(N, local_cap=local_cap, global_cap=global_cap)
        # (requests, share of refused hashes); 1.0: a hash buffer that nobody filled
        for n, refused in ((7, 0.3), (cap_req, 0.0), (60, 0.2), (1, 1.0), (cap_req, 0.01), (33, 1.0), (200, 0.0)):
            nblk = rng.integers(0, 6, size=n)
            off = np.zeros(n + 1, np.int64)
            np.cumsum(nblk * B, out=off[1:])
            total = int(nblk.sum())
            inst = rng.integers(-1, N, size=n).astype(np.int32)
            h = pool[rng.integers(0, len(pool), size=total)]
            bad = rng.random(total) < refused
            h[bad] = rng.integers(0, 2, size=int(bad.sum()), dtype=np.uint64)
            out = dict(instance=T(inst), local_hit=T(np.zeros(n, np.int32)), block_hashes=T(np.append(h, np.uint64(2))))
            ix.commit_batch(T(off), out, also_global=True)
            row = np.repeat(np.arange(n), nblk)
            took = (inst[row] >= 0) & ~bad
            assert ix.status() == (pkg.SMETRIC_ERR_INVALID_ARG if np.any(bad & (inst[row] >= 0)) else pkg.SMETRIC_OK)
            ol.commit(np.bincount(row[took], minlength=n)[inst >= 0], inst[inst >= 0], h[took], also_global=True)
            seen.update(h[took].tolist())
            assert ix.lru_sizes().cpu().numpy().tolist() == [ol.size(i) for i in range(N)] + [ol.size(-1)]
            keys = np.array(sorted(seen), np.uint64)
            m = ix.lookup(T(keys)).cpu().numpy().view(np.uint64)
            for t in ([*range(N)] if local_cap else []) + ([-1] if global_cap else []):
                bit = N if t < 0 else t
                got = keys[(m[:, bit >> 6] >> np.uint64(bit & 63)) & np.uint64(1) == 1]
                assert set(got.tolist()) == set(ol.stamp[t]), (caps, n, t)
    ix.close()
