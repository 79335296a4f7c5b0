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


@pytest.mark.parametrize("n,per,cap", [(7, 30, 1000), (4000, 1000, 30_500_000)])
def test_more_tiles_than_ctas(n, per, cap):
    """Commits on one tier, at the largest with more tiles than the kernels have CTAs; a key's stamp is that of
    its last touch, and the tier keeps the `cap` largest (on the small case the LRU oracle says the same)."""
    N, B, K = 2, 2, 9
    ix = make_index(N, B, 1, cap=2 * K * n * per, max_req=n, max_tok=n * per * B)
    ix.set_lru(cap)
    off = torch.arange(n + 1, device="cuda") * (per * B)
    who = torch.zeros(n, dtype=torch.int32, device="cuda")
    key_of = lambda i: (i + 1) * -7046029254386353131  # noqa: E731  (odd: another key for every i)
    ol = oracle.OracleLRU(N, local_cap=cap)
    stamp = torch.zeros(K * n * per, dtype=torch.int64, device="cuda")
    late = (torch.arange(n * per, device="cuda") // per + 1) * per - torch.arange(n * per, device="cuda") % per  # by request, then deepest first
    for k in range(K):
        first = k * n * per
        i = torch.arange(first, first + n * per, device="cuda")
        if k % 2:  # half of it was there before, some of that evicted since
            i[: n * per // 2] = i[: n * per // 2] * 3 // 5
        h = key_of(i)
        ix.commit_batch(off, dict(instance=who, local_hit=torch.zeros_like(who), block_hashes=h))
        stamp.scatter_reduce_(0, i, late + first, "amax")
        if n < 100:
            ol.commit(np.full(n, per), who.cpu().numpy(), h.cpu().numpy().view(np.uint64), also_global=False)
    ix.check()
    assert ix.lru_sizes().tolist() == [min(cap, int((stamp > 0).sum())), 0, 0]
    least = torch.sort(stamp, descending=True).values[cap - 1]
    held = (ix.lookup(key_of(torch.arange(K * n * per, device="cuda"))).view(torch.int64)[:, 0] & 1) == 1
    assert torch.equal(held, (stamp >= least) & (stamp > 0))
    if n < 100:
        keys = key_of(torch.arange(K * n * per, device="cuda"))[held].cpu().numpy().view(np.uint64)
        assert set(keys.tolist()) == set(ol.stamp[0])
    ix.close()
