"""Cases that time the routing library through its public entry points.

A case is what a router, a replay or a trace study has the library do for one
batch: its path, the batch size, the instances (N), the block size (B), the
mean prompt length and what the traffic looks like.

Traffic, generated on the GPU from the seed (the shapes of synth/traces.py):
  burst  requests drawn from 65,536 concurrent sessions with Zipf(1.1)
         popularity; 95 % of a prompt is the session's cached prefix, which
         the global tier holds, its home instance with probability 0.8 and
         one other instance with probability 0.2. Popular sessions come
         several times in a batch and share their prefix.
  agent  every request is the next turn of a session of its own: one of a few
         system prompts, the session's history (held by its home instance and
         mostly by the global tier) and 256 to 4,096 new tokens. With
         `truncate`, that share of the requests dropped the head of its
         history, so that nothing of it is stored.
Prompt lengths are uniform within two thirds of their mean (a burst of fewer
than 8 requests has them all at the mean). The index holds
random other keys up to a load factor of 0.7.

Every output is an integer and reproducible, so every tolerance is "exact".
"""

import math

import numpy as np
import torch

import paper_2607_08565_gb300 as smetric

DEV = "cuda"
VOCAB = 151936
WEIGHTS = (1, 4, 2)  # load, miss, global fetch
POLICY = dict(c_lin=1000, c_att=1, ttft_d0=400_000_000, ttft_d1=4000, hit_num=9, hit_den=10, rr_base=3)
LAMBDA = (1, 2)
SESSIONS, ZIPF = 65536, 1.1
RING = 8  # batches that a replay case goes through in turn
WINDOW_MS, DAY_MS = 30_000, 4 * 3_600_000
TAG_OTHERS, TAG_EVICTED, TAG_CACHES, TAG_RING = 1, 2, 3, 4  # of the seeds derived from a case's
MAX_TOKENS = 400_000_000  # of a drawn case; the largest listed one has about 790 million


def listed():
    return [
        # One request at a time: an online router that decides on arrival.
        dict(name="route one", path="route", traffic="burst", n=1, N=64, B=32, mean=24000),
        # A router that gets a few requests in host memory and needs the answer there.
        dict(name="host 16", path="host", traffic="agent", n=16, N=16, B=16, mean=6000),
        # The tiny agent trace's batch: 64 sessions, 4 instances, no global tier, hashes wanted for the
        # index's upkeep.
        dict(name="agent 64", path="route", traffic="agent", n=64, N=4, B=16, mean=5000, hashes=True, stored_globally=0.0),
        # A replay step of the medium agent trace: route, commit, drain and LRU eviction on the device.
        dict(name="replay 256", path="commit", traffic="agent", n=256, N=16, B=16, mean=12000, local_cap=200_000),
        # The session-centric policy over a ragged batch on a larger cluster.
        dict(name="policy 777", path="policy", traffic="agent", n=777, N=100, B=32, mean=20000, decide="session"),
        # The long-context coding trace: half the requests truncated, prompts to 110k tokens.
        dict(name="long 1024", path="route", traffic="agent", n=1024, N=32, B=64, mean=66000, hashes=True, truncate=0.5),
        # Loads updated request by request within the batch.
        dict(name="sequential 4096", path="sequential", traffic="burst", n=4096, N=64, B=32, mean=24000),
        # The most instances the index takes, with small blocks.
        dict(name="burst 4099 N=256", path="route", traffic="burst", n=4099, N=256, B=16, mean=24000),
        # The burst trace's batch, on which the throughput is quoted.
        dict(name="burst 8192", path="route", traffic="burst", n=8192, N=64, B=32, mean=24000),
        # The largest batch of the stress sweep.
        dict(name="burst 32768", path="route", traffic="burst", n=32768, N=64, B=32, mean=24000),
        # Index upkeep: a store's prompts hashed and inserted, a third evicted, all looked up.
        dict(name="upkeep 1500", path="upkeep", traffic="agent", n=1500, N=32, B=32, mean=16000),
        # Trace study of a window: sessions linked, reuse broken down, load imbalance per 30 s.
        dict(name="study 8192", path="study", traffic="agent", n=8192, N=32, B=16, mean=12000, turns=8),
    ]


def draw(rng):
    def about(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    path = rng.choice(["route", "route", "route", "route", "host", "commit", "policy", "sequential", "upkeep", "study"])
    c = dict(path=path, traffic=rng.choice(["burst", "agent"]), N=about(4, 256), B=rng.choice([16, 16, 32, 32, 64, 64, 128]), mean=about(3000, 66000))
    most = {"route": 32768, "host": 512, "commit": 1024, "policy": 8192, "sequential": 3000, "upkeep": 2000, "study": 8000}[path]
    limit = {"host": 8_000_000, "commit": 20_000_000, "upkeep": 40_000_000, "study": 80_000_000}.get(path, MAX_TOKENS)
    c["n"] = min(about(64 if path in ("commit", "upkeep", "study") else 1, most), max(1, int(limit / c["mean"])))
    if path in ("commit", "upkeep", "study"):
        c["traffic"] = "agent"
    if path == "route":
        c["hashes"] = rng.random() < 0.4
    if path == "commit":
        c["local_cap"] = about(2000, 200_000) // max(1, c["N"] // 16)
    if path == "policy":
        c["decide"] = rng.choice(["session", "coloc", "bailian", "lmetric"])
    if path == "study":
        c["turns"] = rng.choice([4, 7, 16])
    if c["traffic"] == "agent":
        c["truncate"] = rng.choice([0.0, 0.5])
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------


def _derived(seed, *tags):
    return int(np.random.SeedSequence([int(seed), *tags]).generate_state(1, np.uint64)[0] >> np.uint64(2))


def _generator(seed, *tags):
    return torch.Generator(device=DEV).manual_seed(_derived(seed, *tags))


def _uniform(g, n, lo, hi):
    """n int64 from [lo, hi)."""
    return torch.randint(int(lo), int(hi), (int(n),), generator=g, device=DEV, dtype=torch.int64)


def _keys(g, n):
    return _uniform(g, n, -(1 << 62), 1 << 62)


def _offsets(lens):
    off = torch.zeros(lens.numel() + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(lens, 0, out=off[1:])
    return off


def _text(rows):
    """The tokens of rows of a system prompt, a history and a fresh tail: the
    token at position p of a text is a function of that text's key and p."""
    lens, off = rows["lens"], _offsets(rows["lens"])
    ends = off.cpu().tolist()
    out = torch.empty(ends[-1], dtype=torch.int32, device=DEV)
    r0, n = 0, lens.numel()
    while r0 < n:  # about 64M tokens at a time
        r1 = min(n, max(r0 + 1, int(np.searchsorted(ends, ends[r0] + (1 << 26)))))
        row = torch.repeat_interleave(torch.arange(r0, r1, device=DEV), lens[r0:r1])
        p = torch.arange(ends[r0], ends[r1], device=DEV) - off[row]
        x = torch.where(p < rows["head"][row], rows["head_key"][row], torch.where(p < rows["past"][row], rows["key"][row], rows["tail_key"][row]))
        x = (x + p * 0x5851F42D4C957F2D) * 0x2545F4914F6CDD1D
        x = (x ^ (x >> 32)) * 0x369DEA0F31A53F85
        x = (x ^ (x >> 29)) & 0x7FFFFFFFFFFFFFFF
        out[ends[r0]:ends[r1]] = (x % VOCAB).to(torch.int32)
        r0 = r1
    return out, off


def _head(case):
    """Tokens of an agent's system prompt."""
    return 4096 if case["mean"] >= 12000 else 2048 if case["mean"] >= 4500 else 512


def _burst(case, g):
    n, N, mean = case["n"], case["N"], case["mean"]
    lens = _uniform(g, SESSIONS, mean // 3, 5 * mean // 3 + 1)
    if n < 8:  # a few requests: their time should not hang on the lengths drawn
        lens.fill_(mean)
    key, home = _keys(g, SESSIONS), _uniform(g, SESSIONS, 0, N)
    other = (home + _uniform(g, SESSIONS, 1, max(N, 2))) % N
    in_home = torch.rand(SESSIONS, generator=g, device=DEV) < 0.8
    in_other = torch.rand(SESSIONS, generator=g, device=DEV) < 0.2
    cdf = torch.cumsum(torch.arange(1, SESSIONS + 1, device=DEV, dtype=torch.float64) ** -ZIPF, 0)
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * cdf[-1]
    s = torch.searchsorted(cdf, u, right=True).clamp_(max=SESSIONS - 1)
    past = (lens.double() * 0.95).long()
    rows = dict(lens=lens[s], past=past[s], key=key[s], tail_key=_keys(g, n), head=torch.zeros_like(s), head_key=torch.zeros_like(s))
    d = torch.unique(s)
    stored = dict(lens=past[d], past=past[d], key=key[d], tail_key=key[d], head=torch.zeros_like(d), head_key=torch.zeros_like(d))
    tiers = torch.stack([torch.full_like(d, -1), torch.where(in_home[d], home[d], -2), torch.where(in_other[d], other[d], -2)])
    return rows, stored, tiers


def _agent(case, g):
    n, N, mean, head = case["n"], case["N"], case["mean"], _head(case)
    low, high = max(mean // 3, head + 256), 5 * mean // 3
    lens = (low + (high - low) * (torch.arange(n, device=DEV) + 0.5) / n).long()[torch.randperm(n, generator=g, device=DEV)]
    grown = torch.exp(torch.rand(n, generator=g, device=DEV) * math.log(16.0) + math.log(256.0)).long()
    past = torch.maximum(lens - grown, torch.full_like(lens, head))
    system = _keys(g, 4)[_uniform(g, n, 0, 4)]
    rows = dict(lens=lens, past=past, key=_keys(g, n), tail_key=_keys(g, n), head=torch.full_like(lens, head), head_key=system)
    # an upkeep call brings the prompts that have run, tail and all
    stored = dict(rows, lens=(lens if case["path"] == "upkeep" else past).clone(), tail_key=rows["key"])
    tiers = torch.stack([_uniform(g, n, 0, N), torch.where(torch.rand(n, generator=g, device=DEV) < case.get("stored_globally", 0.9), -1, -2)])
    cut = torch.rand(n, generator=g, device=DEV) < case.get("truncate", 0.0)
    rows["head"] = torch.where(cut, 0, rows["head"])
    rows["past"] = torch.where(cut, 0, rows["past"])
    return rows, stored, tiers


def _window(case, g):
    """A window of a trace in turn waves: request r is turn r // S of session r % S."""
    turns, head, mean = case["turns"], _head(case), case["mean"]
    S = -(-case["n"] // turns)
    per = torch.rand(S, generator=g, device=DEV) * 1.8 + 0.1
    growth = (per * 2 * max(mean - head, 256) / (turns + 1)).long() + 32
    r = torch.arange(case["n"], device=DEV)
    s, t = r % S, r // S
    lens = head + growth[s] * (t + 1)
    cut = torch.rand(case["n"], generator=g, device=DEV) < case.get("truncate", 0.0)
    key, system, own = _keys(g, S), _keys(g, 4)[_uniform(g, S, 0, 4)], _keys(g, case["n"])
    rows = dict(lens=torch.where(cut, lens * 3 // 4, lens), past=torch.where(cut, 0, lens), key=key[s], tail_key=own, head=torch.where(cut, 0, head), head_key=system[s])
    start = torch.sort(_uniform(g, case["n"], 0, DAY_MS - 600_000)).values
    ran = torch.exp(torch.randn(case["n"], generator=g, device=DEV) + math.log(8000.0)).long().clamp_(max=600_000)
    extra = dict(users=s.clone(), turns=t.int(), sys_blocks=torch.where(cut, 0, head // case["B"]).int(), instance=_uniform(g, case["n"], 0, case["N"]).int(), start=start, end=start + ran)
    return rows, extra


def _loads(case, g):
    N = case["N"]
    d = dict(load=_uniform(g, N, 0, 2_000_001))
    d["requests"] = _uniform(g, N, 1, 65)
    d["tpot"] = torch.where(torch.rand(N, generator=g, device=DEV) < 0.25, 1 << 60, _uniform(g, N, 10**7, 10**9))
    return d


def _inputs(case, seed):
    g = _generator(seed, case["n"], case["N"], case["B"], case["mean"])
    if case["path"] == "study":
        rows, extra = _window(case, g)
        tokens, offsets = _text(rows)
        return dict(extra, tokens=tokens, offsets=offsets)
    rows, stored, tiers = (_burst if case["traffic"] == "burst" else _agent)(case, g)
    d = _loads(case, g)
    d["tokens"], d["offsets"] = _text(rows)
    d["stored_tokens"], d["stored_offsets"] = _text(stored)
    d["stored_tiers"] = tiers
    n = case["n"]
    d["turn"] = (torch.rand(n, generator=g, device=DEV) >= 0.1).int()
    d["expected"] = rows["past"].clone()
    return d


def _blocks(offsets, B):
    return (offsets[1:] - offsets[:-1]) // B


def _most_blocks(case):
    """Room for a batch's block hashes, as a program keeps it for any batch of this size."""
    return max(1, case["n"] * (5 * case["mean"] // 3 + 1) // case["B"])


def _pairs(keys, offsets, tiers, B):
    """(key, tier) pairs of stored prompts' block hashes; a tier row of -2 holds nothing."""
    t = torch.repeat_interleave(tiers, _blocks(offsets, B), dim=1)
    keep = t > -2
    return torch.cat([keys[k] for k in keep]), t[keep].int()


def _shape(case, tokens):
    # session blocks: the system prompt and one more, or the first block
    S = _head(case) // case["B"] + 1 if case["traffic"] == "agent" else 1
    return dict(num_instances=case["N"], block_size=case["B"], session_blocks=S, max_batch_requests=case["n"], max_batch_tokens=tokens)


def _outputs(n, *names, device=DEV):
    kinds = dict(session_key=torch.int64)
    return {k: torch.zeros(n, dtype=kinds.get(k, torch.int32), device=device) for k in names}


ROUTED = ("instance", "local_hit", "global_hit", "session_key")


def _index(case, d, seed, **more):
    """An index that holds the stored prompts, and other keys up to 0.7 of its slots."""
    B, most = case["B"], max(d["tokens"].numel(), d["stored_tokens"].numel())
    n_stored = int(_blocks(d["stored_offsets"], B).sum())
    slots = 1 << 26 if case["n"] >= 4096 else 1 << 24
    slots = max(slots, int(1.6 * n_stored))
    c = dict(_shape(case, most), max_batch_requests=max(case["n"], d["stored_offsets"].numel() - 1))
    ix = smetric.SMetricIndex(capacity_slots=slots, **c, **more)
    hashes, _ = ix.block_hashes(d["stored_tokens"], d["stored_offsets"])
    keys, tiers = _pairs(hashes.view(torch.int64)[:n_stored], d["stored_offsets"], d["stored_tiers"], B)
    ix.insert(keys, tiers)
    g = _generator(seed, TAG_OTHERS)
    other = int(0.7 * slots) - n_stored
    if other > 0:
        ix.insert(_keys(g, other) * 2 + 5, _uniform(g, other, -1, case["N"]).int())
    ix.check()
    return ix


def prepare(case, seed):
    case = dict(case)
    if case["path"] == "study":
        return _prepare_study(case, seed)
    if case["path"] == "commit":
        return _prepare_commit(case, seed)
    d = _inputs(case, seed)
    n, B = case["n"], case["B"]
    s = dict(path=case["path"], decide=case.get("decide"), tokens=d["tokens"], offsets=d["offsets"], load=d["load"])
    if case["path"] == "upkeep":
        n_blocks = int(_blocks(d["stored_offsets"], B).sum())
        ix = smetric.SMetricIndex(capacity_slots=max(1 << 16, 3 * n_blocks), **_shape(case, d["stored_tokens"].numel()))
        hashes, _ = ix.block_hashes(d["stored_tokens"], d["stored_offsets"])
        keys, tiers = _pairs(hashes.view(torch.int64)[:n_blocks], d["stored_offsets"], d["stored_tiers"], B)
        out = torch.rand(keys.numel(), generator=_generator(seed, TAG_EVICTED), device=DEV) < 1 / 3
        s.update(tokens=d["stored_tokens"], offsets=d["stored_offsets"], n_blocks=n_blocks, ix=ix)
        s.update(keys=keys, tiers=tiers, evict_keys=keys[out], evict_tiers=tiers[out])
        return s
    s["ix"] = _index(case, d, seed, host_staging=case["path"] == "host")
    if case["path"] == "host":
        for k in ("tokens", "offsets", "load"):
            s[k] = s[k].cpu().pin_memory()
        s["out"] = {k: v.pin_memory() for k, v in _outputs(n, *ROUTED, device="cpu").items()}
    elif case["path"] == "policy":
        s.update(queued=d["load"] * 256, turn=d["turn"], expected=d["expected"], tpot=d["tpot"], requests=d["requests"])
        s["out"] = _outputs(n, *ROUTED, "stick")
    elif case["path"] == "route":
        s["out"] = _outputs(n, *ROUTED)
        if case.get("hashes"):
            s["out"]["block_hashes"] = torch.zeros(_most_blocks(case), dtype=torch.int64, device=DEV)
    return s


def _prepare_commit(case, seed):
    """Full caches, and RING batches of other sessions that a pass takes in turn."""
    n, N, B, cap = case["n"], case["N"], case["B"], case["local_cap"]
    ring = [_inputs(case, _derived(seed, TAG_RING, k)) for k in range(RING)]
    most = max(max(d["tokens"].numel(), d["stored_tokens"].numel()) for d in ring)
    live = 2 * N * cap + 2 * sum(int(_blocks(d["offsets"], B).sum()) for d in ring)
    ix = smetric.SMetricIndex(capacity_slots=max(1 << 16, int(live / 0.6)), **_shape(case, most))
    ix.set_lru(local_cap=cap)
    # earlier traffic: every instance's cache full of other blocks
    g = _generator(seed, TAG_CACHES)
    per = min(max(1, most // B // n), cap)
    off = torch.arange(n + 1, device=DEV, dtype=torch.int64) * (per * B)
    for first in range(0, N * -(-cap // per), n):
        who = ((torch.arange(n, device=DEV) + first) % N).int()
        earlier = dict(instance=who, local_hit=torch.zeros_like(who), block_hashes=_keys(g, n * per) * 2 + 5)
        ix.commit_batch(off, earlier, also_global=True)
    # the sessions' earlier turns
    for d in ring:
        hashes, _ = ix.block_hashes(d["stored_tokens"], d["stored_offsets"])
        who = d["stored_tiers"][0].int()
        ix.commit_batch(d["stored_offsets"], dict(instance=who, local_hit=torch.zeros_like(who), block_hashes=hashes), also_global=True)
    ix.check()
    out = dict(_outputs(n, *ROUTED), block_hashes=torch.zeros(_most_blocks(case), dtype=torch.int64, device=DEV))
    return dict(path="commit", ix=ix, ring=[(d["tokens"], d["offsets"]) for d in ring], load=ring[0]["load"], out=out, at=0)


def _prepare_study(case, seed):
    d = _inputs(case, seed)
    tokens = d["tokens"].numel()
    ix = smetric.SMetricIndex(capacity_slots=1 << 16, **_shape(case, tokens))
    windows = DAY_MS // WINDOW_MS
    need = smetric.smetric_reuse_workspace_bytes(tokens // case["B"])
    return dict(
        d, path="study", ix=ix, windows=windows, reuse_space=torch.empty(need, dtype=torch.uint8, device=DEV),
        imbalance_space=torch.empty(smetric.smetric_imbalance_workspace_bytes(windows, case["N"]) // 8, dtype=torch.int64, device=DEV))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------


def _signed(out):
    return {k: v.view(torch.int64) if v.dtype == torch.uint64 else v for k, v in out.items()}


def run(state):
    s, ix = state, state["ix"]
    path = s["path"]
    if path == "route":
        return ix.route_batch(s["tokens"], s["offsets"], s["load"], WEIGHTS, out=s["out"])
    if path == "host":
        o = s["out"]
        rc = smetric.smetric_route_batch_host(ix.handle, s["tokens"], s["tokens"].numel(), s["offsets"], s["offsets"].numel() - 1, s["load"], WEIGHTS,
                                              o["instance"], o["local_hit"], o["global_hit"], o["session_key"])
        if rc != smetric.SMETRIC_OK:
            raise smetric.SmetricError(rc, "smetric_route_batch_host")
        return o
    if path == "sequential":
        return _signed(ix.route_batch_sequential(s["tokens"], s["offsets"], s["load"], WEIGHTS))
    if path == "policy":
        if s["decide"] == "session":
            return ix.route_batch_policy(s["tokens"], s["offsets"], s["queued"], s["turn"], s["expected"], POLICY, out=s["out"])
        if s["decide"] == "coloc":
            return _signed(ix.route_batch_policy_coloc(s["tokens"], s["offsets"], s["queued"], s["tpot"], s["requests"], s["turn"], s["expected"], POLICY))
        scorer = smetric.SMETRIC_SCORER_BAILIAN if s["decide"] == "bailian" else smetric.SMETRIC_SCORER_LMETRIC
        return _signed(ix.route_batch_baseline(s["tokens"], s["offsets"], scorer, s["load"], s["requests"], LAMBDA))
    if path == "commit":
        tokens, offsets = s["ring"][s["at"]]
        s["at"] = (s["at"] + 1) % len(s["ring"])
        o = s["out"]
        smetric.smetric_route_commit_batch(ix.handle, tokens, tokens.numel(), offsets, offsets.numel() - 1, s["load"], WEIGHTS, o["instance"], o["local_hit"],
                                           o["global_hit"], o["session_key"], o["block_hashes"], o["block_hashes"].numel(), smetric.SMETRIC_COMMIT_GLOBAL)
        return dict(o, load=s["load"])
    if path == "upkeep":
        hashes, session = ix.block_hashes(s["tokens"], s["offsets"])
        ix.insert(s["keys"], s["tiers"])
        ix.evict(s["evict_keys"], s["evict_tiers"])
        keys = hashes[: s["n_blocks"]]
        return dict(keys=keys.view(torch.int64), session_key=session.view(torch.int64), masks=ix.lookup(keys).view(torch.int64))
    parent, session = ix.link_sessions(s["tokens"], s["offsets"], s["users"], s["turns"])
    reuse = ix.reuse_breakdown(s["tokens"], s["offsets"], session, s["sys_blocks"], workspace=s["reuse_space"])
    load = ix.window_imbalance(s["instance"], s["start"], s["end"], WINDOW_MS, s["windows"], workspace=s["imbalance_space"])
    return dict(parent=parent, session=session, reuse=reuse, load=load)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------


def work(case):
    """Bytes: the tokens and offsets read, the index entries that the prefix
    match has to see (a prefix that several requests share once), block hashes
    where the caller gets them, and the outputs. There is no floating-point
    arithmetic on this path."""
    n, N, B, mean = case["n"], case["N"], case["B"], case["mean"]
    W = (N + 1 + 63) // 64
    blocks = n * mean / B
    tokens = 4.0 * n * mean + 8 * (n + 1)
    if case["path"] == "study":
        # link and reuse each read the window's tokens; the imbalance reads its requests
        return dict(bytes=2 * tokens + 16 * blocks + n * (12 + 8 + 8 + 16 + 20) + DAY_MS // WINDOW_MS * (8 * N + 20), flops=0)
    if case["path"] == "upkeep":
        pairs = 1.9 * blocks
        return dict(bytes=tokens + pairs * 4 / 3 * (12 + 8 + 8 * W) + blocks * (8 + 8 + 8 + 16 * W), flops=0)
    if case["traffic"] == "burst":
        p = np.arange(1, SESSIONS + 1) ** -ZIPF
        seen = float((1 - (1 - p / p.sum()) ** n).sum())
        probed = 0.95 * seen * mean / B + n
    else:
        probed = (1 - case.get("truncate", 0.0)) * (blocks - n * 1386.0 / B) + n
    total = tokens + probed * (8 + 8 * W) + 20.0 * n + 8 * N
    if case["path"] == "policy":
        total += 16.0 * n
    if case.get("hashes") or case["path"] == "commit":
        total += 8 * blocks
    if case["path"] == "commit":
        # each new block enters two tiers and leaves one; each touch reorders its tier's records
        total += 2 * blocks * (8 + 8 * W) + 16 * blocks
    return dict(bytes=total, flops=0)


def tolerance(case):
    return "exact"


# ---------------------------------------------------------------------------
# the same in plain torch, on 64-bit integers
# ---------------------------------------------------------------------------


def _s64(x):
    x &= (1 << 64) - 1
    return x - (1 << 64) if x >> 63 else x


GAMMA = 0x9E3779B97F4A7C15
M1, M2 = _s64(0xBF58476D1CE4E5B9), _s64(0x94D049BB133111EB)


def _shr(x, k):
    return (x >> k) & ((1 << (64 - k)) - 1)


def _mix(z):
    z = (z ^ _shr(z, 30)) * M1
    z = (z ^ _shr(z, 27)) * M2
    return z ^ _shr(z, 31)


def _mix_of(x):
    return int(_mix(torch.tensor([_s64(x)]))[0])


def _hash(tokens, offsets, B):
    """Every full block's chain hash, request after request."""
    nb = _blocks(offsets, B)
    first = _offsets(nb)
    row = torch.repeat_interleave(torch.arange(nb.numel(), device=DEV), nb)
    at = offsets[row] + (torch.arange(row.numel(), device=DEV) - first[row]) * B
    d = torch.full((row.numel(),), _mix_of(B), dtype=torch.int64, device=DEV)
    for k in range(0, B, 2):
        d = _mix(d ^ (tokens[at + k].long() & 0xFFFFFFFF | tokens[at + k + 1].long() << 32))
    order = torch.argsort(nb, descending=True)
    longest = np.sort(nb.cpu().numpy())
    out = torch.empty_like(d)
    h = torch.full((nb.numel(),), _mix_of(GAMMA), dtype=torch.int64, device=DEV)
    for b in range(int(longest[-1])):
        m = nb.numel() - int(np.searchsorted(longest, b, side="right"))
        i = first[:-1][order[:m]] + b
        x = _mix((h[:m] + _s64(GAMMA)) ^ d[i])
        h[:m] = torch.where((x == 0) | (x == 1), x | 2, x)
        out[i] = h[:m]
    return out, first, row


def _session_keys(H, first, S):
    nb = first[1:] - first[:-1]
    at = first[:-1] + torch.clamp(nb, max=S) - 1
    return torch.where(nb > 0, H[at.clamp(min=0)], 0)


def _masks(query, keys, tiers, N):
    """Tier masks [len(query), W] of keys in a store of (key, tier) pairs."""
    W = (N + 1 + 63) // 64
    known, where = torch.unique(keys, return_inverse=True)
    bit = torch.where(tiers < 0, N, tiers.long())
    pair = torch.unique(where * (N + 1) + bit)  # a pair counts once
    m = torch.zeros((known.numel() + 1, W), dtype=torch.int64, device=DEV)
    bit = pair % (N + 1)
    m.view(-1).index_add_(0, pair // (N + 1) * W + bit // 64, torch.ones_like(pair) << (bit % 64))
    at = torch.searchsorted(known, query).clamp_(max=known.numel() - 1)
    return m[torch.where(known[at] == query, at, known.numel())]


def _runs(masks, first, row, N):
    """[n, N + 1]: the leading blocks that each tier holds (the global one last)."""
    nb = first[1:] - first[:-1]
    pos = torch.arange(row.numel(), device=DEV) - first[row]
    out = torch.empty((nb.numel(), N + 1), dtype=torch.int64, device=DEV)
    for t in range(N + 1):
        gone = (masks[:, t // 64] >> (t % 64)) & 1 == 0
        out[:, t] = nb.scatter_reduce(0, row[gone], pos[gone], "amin")
    return out


def _first_min(x):
    low = x.min(1, keepdim=True).values
    return torch.where(x == low, torch.arange(x.shape[1], device=DEV), x.shape[1]).min(1).values


def _pick(x, i):
    return x.gather(1, i[:, None])[:, 0]


def _padded(H, case):
    out = torch.zeros(_most_blocks(case), dtype=torch.int64, device=DEV)
    out[: H.numel()] = H
    return out


def exact(case, seed):
    d = _inputs(case, _derived(seed, TAG_RING, 0) if case["path"] == "commit" else seed)
    N, B, n = case["N"], case["B"], case["n"]
    S = _shape(case, 0)["session_blocks"]
    if case["path"] == "study":
        return _exact_study(case, d)
    if case["path"] == "upkeep":
        H, first, _ = _hash(d["stored_tokens"], d["stored_offsets"], B)
        keys, tiers = _pairs(H, d["stored_offsets"], d["stored_tiers"], B)
        out = torch.rand(keys.numel(), generator=_generator(seed, TAG_EVICTED), device=DEV) < 1 / 3
        # a pair that several prompts have is gone when one of them is evicted
        pair = torch.unique(keys, return_inverse=True)[1] * (N + 1) + torch.where(tiers < 0, N, tiers.long())
        kept = ~torch.isin(pair, pair[out])
        return dict(keys=H, session_key=_session_keys(H, first, S), masks=_masks(H, keys[kept], tiers[kept], N))
    H, first, row = _hash(d["tokens"], d["offsets"], B)
    session_key = _session_keys(H, first, S)
    if case["path"] == "commit":  # the rest depends on what earlier commits left in the caches
        return dict(instance=None, local_hit=None, global_hit=None, session_key=session_key, block_hashes=_padded(H, case), load=None)
    stored, _, _ = _hash(d["stored_tokens"], d["stored_offsets"], B)
    keys, tiers = _pairs(stored, d["stored_offsets"], d["stored_tiers"], B)
    runs = _runs(_masks(H, keys, tiers, N), first, row, N)
    c, run_g = runs[:, :N], runs[:, N:]
    L = (d["offsets"][1:] - d["offsets"][:-1])[:, None]
    reach = torch.maximum(c, run_g)
    load = d["load"][None, :]
    rest = WEIGHTS[1] * (L - B * reach) + WEIGHTS[2] * B * (reach - c)
    more = {}
    if case["path"] == "sequential":
        q, rest_h, new = d["load"].cpu().numpy().copy(), rest.cpu().numpy(), (L - B * c).cpu().numpy()
        to = np.empty(n, np.int64)
        for r in range(n):
            to[r] = np.argmin(WEIGHTS[0] * q + rest_h[r])
            q[to[r]] += new[r, to[r]]
        to = torch.from_numpy(to).to(DEV)
        more["load_after"] = torch.from_numpy(q).to(DEV)
    elif case["path"] == "policy":
        to, more = _decide(case, d, c, L)
    else:
        to = _first_min(WEIGHTS[0] * load + rest)
    hit = _pick(c, to)
    out = dict(instance=to.int(), local_hit=(B * hit).int(), global_hit=(B * (torch.maximum(hit, run_g[:, 0]) - hit)).int(), session_key=session_key, **more)
    if case.get("hashes"):
        out["block_hashes"] = _padded(H, case)
    return out


def _decide(case, d, c, L):
    """The policies' choices; their products stay below 2^63 on these inputs."""
    N, B, n = case["N"], case["B"], case["n"]
    if case["decide"] in ("bailian", "lmetric"):
        requests = d["requests"][None, :]
        if case["decide"] == "lmetric":
            return _first_min((d["load"][None, :] + L - B * c) * requests), {}
        num, den = LAMBDA
        return _first_min((den - num) * requests * L + num * (L - B * c) * requests.max()), {}
    new = L - B * c
    cost = 2 * POLICY["c_lin"] * new + POLICY["c_att"] * new * (2 * L - new)
    est = 2 * 256 * d["load"][None, :] + cost
    meets = est <= 2 * (POLICY["ttft_d0"] + POLICY["ttft_d1"] * L)
    prev = _first_min(-c)
    cached = B * _pick(c, prev) * POLICY["hit_den"] > POLICY["hit_num"] * d["expected"]
    start = (POLICY["rr_base"] + torch.arange(n, device=DEV)) % N
    turn = (start[:, None] + torch.arange(N, device=DEV)[None, :]) % N  # scan order
    if case["decide"] == "session":
        stick = (d["turn"] != 0) & cached & (_pick(meets, prev) | ~meets.any(1))
        score = est
    else:
        fits = cost <= 2 * d["tpot"][None, :]
        fits |= ~fits.any(1, keepdim=True)
        stick = (d["turn"] != 0) & cached & _pick(meets, prev) & _pick(fits, prev)
        score = torch.where(fits, est * d["requests"][None, :], (1 << 63) - 1)
    balanced = _pick(turn, _first_min(score.gather(1, turn)))
    return torch.where(stick, prev, balanced), dict(stick=stick.int())


def _exact_study(case, d):
    n, N, B = case["n"], case["N"], case["B"]
    H, first, row = _hash(d["tokens"], d["offsets"], B)
    nb = first[1:] - first[:-1]
    pos = torch.arange(row.numel(), device=DEV) - first[row]
    # a user is a session here, so a parent is the same user's previous turn where it is a prefix
    r = torch.arange(n, device=DEV)
    S = -(-n // case["turns"])
    p = (r - S).clamp(min=0)
    last = torch.where(nb[p] > 0, H[(first[:-1][p] + nb[p] - 1).clamp(min=0)], 0)
    mine = torch.where(nb[p] > 0, H[(first[:-1] + nb[p] - 1).clamp(max=H.numel() - 1)], 0)
    parent = torch.where((r >= S) & (nb[p] <= nb) & (last == mine), p, -1)
    session = torch.where(parent < 0, r, parent)
    for _ in range(case["turns"]):
        session = session[session]
    # earliest request holding each block
    known, where = torch.unique(H, return_inverse=True)
    holder = torch.full((known.numel(),), n, dtype=torch.int64, device=DEV).scatter_reduce(0, where, row, "amin")[where]
    hit = nb.scatter_reduce(0, row[holder >= row], pos[holder >= row], "amin")
    within = pos < hit[row]
    sys = within & (pos < d["sys_blocks"].long()[row])
    intra = within & ~sys & (session[holder.clamp(max=n - 1)] == session[row])
    count = lambda m: torch.zeros(n, dtype=torch.int64, device=DEV).index_add_(0, row, m.long()).int()  # noqa: E731
    reuse = dict(hit=hit.int(), sys=count(sys), intra=count(intra), inter=count(within & ~sys & ~intra))
    cells = torch.zeros(DAY_MS // WINDOW_MS * N, dtype=torch.int64, device=DEV)
    for k in range(600_000 // WINDOW_MS + 1):  # the k-th window that a request runs in
        w = d["start"] // WINDOW_MS + k
        ran = torch.minimum(d["end"], (w + 1) * WINDOW_MS) - torch.maximum(d["start"], w * WINDOW_MS)
        on = (ran > 0) & (w < DAY_MS // WINDOW_MS)
        cells.index_add_(0, (w * N + d["instance"])[on], ran[on])
    cells = cells.view(-1, N)
    load = dict(max=cells.max(1).values, argmax=_first_min(-cells).int(), sum=cells.sum(1))
    return dict(parent=parent.int(), session=session.int(), reuse=reuse, load=load)
