"""The chain kernel's shared-memory ring and the walk's own tails, at the sizes
where their work splits change, against the oracle (every value exact)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2607_08565_gb300 as pkg
from gpu_util import T, assert_outputs_equal, gpu_hashes, gpu_route, make_index, populate_both
from pins import GAMMA, M64, _py_mix64, py_mix64_inverse
from synth.traces import pack

pytestmark = pytest.mark.gpu


def _tokens(rng, n):
    return rng.integers(0, 151936, size=int(n), dtype=np.int32)


@pytest.mark.parametrize("N,S,hashes", [(5, 1, True), (64, 3, False), (130, 400, True), (256, 40, False)])
def test_members_with_short_and_long_tails(N, S, hashes):
    """More than four requests an SM, so that members' short tails are chained
    by the walk: tails of 0 to 257 blocks (256 is the longest it takes, a
    quarter of the prompt at most), some of them stored, session keys inside
    the shared prefix and in the tail."""
    rng = np.random.default_rng(N)
    B = 2
    bases = [_tokens(rng, B * nb) for nb in (1, 4, 33, 64, 200, 1100, 1101)]
    tails = [_tokens(rng, B * 260) for _ in range(3)]
    reqs = []
    for base in bases:
        nb = len(base) // B
        reqs.append(base)
        for t in (0, 1, 7, 8, 31, 32, 33, 65, 255, 256, 257):
            for k in (nb, max(1, nb - 1), max(1, nb // 2)):
                reqs.append(np.concatenate([base[:k * B], tails[t % 3][:t * B + t % 2]]))
    while len(reqs) < 900:
        base = bases[int(rng.integers(len(bases)))]
        k = int(rng.integers(1, len(base) // B + 1))
        reqs.append(np.concatenate([base[:k * B], _tokens(rng, rng.integers(0, 90))]))
    reqs += [np.zeros(0, np.int32), bases[0][:1]]
    reqs = [reqs[i] for i in rng.permutation(len(reqs))]
    stored = {t: [reqs[int(rng.integers(len(reqs)))] for _ in range(2)] for t in range(-1, N)}
    stored[-1] += [np.concatenate([bases[5], tails[1][:B * 200]]), np.concatenate([bases[6], tails[0]])]
    stored[0] += [np.concatenate([bases[5], tails[1][:B * 40]])]
    ix = make_index(N, B, S, cap=1 << 18)
    ox = oracle.OracleIndex(N)
    populate_both(ix, ox, stored, B)
    tok, off = pack(reqs)
    for load in (np.zeros(N, np.int64), rng.integers(0, 2000, size=N)):
        g = gpu_route(ix, tok, off, load, (1, 4, 2), want_hashes=hashes)
        o = ox.route_batch(B, S, 0, tok, off, load, 1, 4, 2, want_hashes=hashes)
        assert_outputs_equal(g, o, ctx=f"N={N}")
    assert (g["global_hit"] > 0).any() and (g["local_hit"] > 0).any()
    ix.close()


@pytest.mark.parametrize("n", [600, 612, 4800, 20000, 32768, 32769, 80000])
def test_requests_per_lane_and_per_round(n):
    """Batches around the numbers of requests an SM takes: one chain warp, four,
    several requests a lane (some empty), the last size whose requests are dealt
    out by the group stage, more than one round a CTA."""
    rng = np.random.default_rng(n)
    B, N = 2, 3
    lens = rng.integers(0, 3 * B, size=n)
    lens[rng.integers(0, n, size=40)] = rng.integers(100, 700, size=40)
    pool = _tokens(rng, 701)  # most requests share their leading blocks with others
    off = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    tok = np.concatenate([pool[:L] for L in lens]).astype(np.int32)
    own = rng.random(n) < 0.3
    for r in np.nonzero(own)[0]:
        tok[off[r]:off[r + 1]] = _tokens(rng, lens[r])
    ix = make_index(N, B, 2, cap=1 << 16, max_req=n, max_tok=len(tok))
    ox = oracle.OracleIndex(N)
    populate_both(ix, ox, {-1: [pool], 1: [pool[:301]], 2: [pool[:64], tok[off[5]:off[6]]]}, B)
    load = rng.integers(0, 20, size=N)
    g = gpu_route(ix, tok, off, load, (1, 4, 2))
    o = ox.route_batch(B, 2, 0, tok, off, load, 1, 4, 2, want_hashes=True)
    assert_outputs_equal(g, o, ctx=f"n={n}")
    hb, sk = gpu_hashes(ix, tok, off)
    assert np.array_equal(hb, o["block_hashes"]) and np.array_equal(sk, o["session_key"])
    ix.close()


@pytest.mark.parametrize("at", [1, 31, 32, 63, 64, 300])
def test_sentinel_in_the_middle_of_a_chain(at):
    """A chain value of 0 or 1 at a block inside a ring slot: the chain goes on
    from the remapped value."""
    rng = np.random.default_rng(at)
    for target in (0, 1):
        head = _tokens(rng, 2 * at)
        h = int(oracle.block_hashes(head, 2, 0)[-1])
        d = py_mix64_inverse(target) ^ ((h + GAMMA) & M64)
        w = py_mix64_inverse(d) ^ _py_mix64(2)
        block = np.array([w & 0xFFFFFFFF, w >> 32], dtype=np.uint32).view(np.int32)
        t = np.concatenate([head, block, _tokens(rng, 150)])
        reqs = [t, _tokens(rng, 500), t[:2 * at + 2], head]
        tok, off = pack(reqs)
        ix = make_index(4, 2, 1)
        ox = oracle.OracleIndex(4)
        populate_both(ix, ox, {-1: [t], 2: [t[:2 * at + 40]]}, 2)
        g = gpu_route(ix, tok, off, np.zeros(4), (1, 4, 2))
        o = ox.route_batch(2, 1, 0, tok, off, np.zeros(4, np.int64), 1, 4, 2, want_hashes=True)
        assert int(o["block_hashes"][at]) == 2 + target
        assert_outputs_equal(g, o, ctx=f"sentinel at {at}")
        ix.close()


@pytest.mark.parametrize("more", [0, 1, 31, 33, 5000])
@pytest.mark.parametrize("phase", [0, 1, 2, 3])
def test_hashes_of_more_than_32_requests_an_sm(more, phase):
    """Hash-only calls on both sides of 32 requests an SM, where a thread per
    request takes over: lengths around its four blocks an access, hash buffers
    in every 32-byte phase, a chain value of 0 and of 1 on the way."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, B, S = 32 * sms + more, 2, 9
    rng = np.random.default_rng(10 * more + phase)
    reqs = [_tokens(rng, k) for k in np.minimum(rng.integers(0, 50, size=n), rng.integers(0, 50, size=n))]
    reqs[7], reqs[n - 1] = _tokens(rng, 2 * 1300 + 1), _tokens(rng, 2 * 677)
    for target in (0, 1):
        head = _tokens(rng, 2 * (18 + target))
        d = py_mix64_inverse(target) ^ ((int(oracle.block_hashes(head, 2, 0)[-1]) + GAMMA) & M64)
        w = py_mix64_inverse(d) ^ _py_mix64(2)
        block = np.array([w & 0xFFFFFFFF, w >> 32], dtype=np.uint32).view(np.int32)
        reqs[100 + target] = np.concatenate([head, block, _tokens(rng, 41)])
    tok, off = pack(reqs)
    ix = make_index(4, B, S, max_req=n, max_tok=len(tok))
    o = oracle.OracleIndex(4).route_batch(B, S, 0, tok, off, np.zeros(4, np.int64), 1, 4, 2, want_hashes=True,
                                          n_threads=8)
    nb = len(o["block_hashes"])
    cap = len(tok) // B
    buf = torch.full((cap + 8,), -1, dtype=torch.int64, device="cuda")
    sk = torch.empty(n, dtype=torch.int64, device="cuda")
    pkg.smetric_block_hashes(ix.handle, T(tok), len(tok), T(off), n, sk, buf[phase:], cap, None)
    ix.check()
    h = buf.cpu().numpy().view(np.uint64)
    assert np.array_equal(h[phase:phase + nb], o["block_hashes"])
    assert np.array_equal(sk.cpu().numpy().view(np.uint64), o["session_key"])
    assert (h[:phase] == 2 ** 64 - 1).all() and (h[phase + nb:] == 2 ** 64 - 1).all()
    assert {2, 3} <= set(h.tolist())
    ix.close()


@pytest.mark.parametrize("N", [1, 32, 33, 65, 128, 129, 256])
@pytest.mark.parametrize("n", [1, 11, 12, 13, 37, 301])
def test_sequential_stages_and_cost_widths(N, n):
    """Batches around the stages of the sequential decision, instance counts
    around its instances per lane, equal costs (the lowest instance), and
    costs on both sides of 2^55, where the reductions change."""
    rng = np.random.default_rng(1000 * N + n)
    B = 4
    pool = _tokens(rng, 400)
    reqs = [np.concatenate([pool[:int(rng.integers(0, 300))], _tokens(rng, rng.integers(0, 40))]) for _ in range(n)]
    ix = make_index(N, B, 2)
    ox = oracle.OracleIndex(N)
    populate_both(ix, ox, {t: [pool[:int(rng.integers(0, 400))]] for t in range(-1, min(N, 9))}, B)
    tok, off = pack(reqs)
    same = np.full(N, 7)
    for w, load in (((1, 4, 2), same), ((0, 0, 0), same), ((1, 4, 2), rng.integers(0, 300, size=N)),
                    ((2 ** 20, 2 ** 20, 1), (1 << 40) - rng.integers(0, 500, size=N)),
                    ((2 ** 20, 3, 2 ** 20), np.full(N, 1 << 40)), ((2 ** 15, 4, 2), np.full(N, (1 << 40) - 1)),
                    ((2 ** 15 - 1, 4, 2), np.full(N, (1 << 40) - 1))):
        load = np.asarray(load, np.int64)
        out = ix.route_batch_sequential(T(tok), T(off), T(load), w)
        ix.check()
        o = ox.route_batch_sequential(B, 2, 0, tok, off, load, *w)
        g = {k: v.cpu().numpy() for k, v in out.items()}
        assert_outputs_equal(g, o, fields=("instance", "local_hit", "global_hit", "session_key", "load_after"),
                             ctx=f"N={N} n={n} w={w}")
    ix.close()


@pytest.mark.parametrize("n", [8191, 8192, 8193, 16385, 1100000])
def test_offsets_scanned_and_checked_in_stretches(n):
    """Batches around the requests that one CTA of the offset scan takes (and one
    past 128 times that): hashes equal the oracle's, and a bad offset or length
    in any stretch makes the batch invalid."""
    rng = np.random.default_rng(n)
    B = 2
    lens = rng.integers(0, 4, size=n)
    off = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=off[1:])
    tok = _tokens(rng, off[-1])
    ix = make_index(2, B, 1, max_req=n, max_tok=len(tok))
    hb, sk = gpu_hashes(ix, tok, off)
    o = oracle.OracleIndex(2).route_batch(B, 1, 0, tok, off, np.zeros(2, np.int64), 1, 4, 2, want_hashes=True,
                                          n_threads=8)
    assert np.array_equal(hb, o["block_hashes"]) and np.array_equal(sk, o["session_key"])
    for at in (1, n // 2, n - 1):
        bad = off.copy()
        bad[at] = len(tok) + 1 if at % 2 else -1
        d_sk = torch.full((n,), 5, dtype=torch.int64, device="cuda")
        d_h = torch.zeros(max(1, len(tok) // B), dtype=torch.int64, device="cuda")
        pkg.smetric_block_hashes(ix.handle, T(tok), len(tok), T(bad), n, d_sk, d_h, d_h.numel(), None)
        assert ix.status() == pkg.SMETRIC_ERR_INVALID_ARG
        assert not d_sk.any()
    ix.close()
