"""smetric_route_batch_host on both sides of the size where batches stop going
through the index's pinned buffer: outputs equal the device path's, and a
latched error is returned and cleared, from pageable and pinned arrays."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2607_08565_gb300 as pkg
from gpu_util import T, gpu_route, make_index
from synth.traces import pack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2047, 2048, 2049, 5000])
@pytest.mark.parametrize("pinned", [False, True])
def test_host_route_sizes(n, pinned):
    rng = np.random.default_rng(n)
    N, B = 7, 2
    pool = rng.integers(0, 151936, size=200, dtype=np.int32)
    reqs = [np.concatenate([pool[:int(rng.integers(0, 200))], rng.integers(0, 99, size=3, dtype=np.int32)])
            for _ in range(n)]
    tok, off = pack(reqs)
    load = rng.integers(0, 300, size=N).astype(np.int64)
    ix = make_index(N, B, 2, max_req=n, max_tok=max(len(tok), 400), host_staging=True)
    hb, _ = ix.block_hashes(T(pool), T(np.array([0, 200], np.int64)))
    ix.insert(hb, T(np.arange(100, dtype=np.int32) % (N + 1) - 1))
    want = gpu_route(ix, tok, off, load, (1, 4, 2), want_hashes=False)

    def host(a):
        t = torch.from_numpy(np.ascontiguousarray(a))
        return t.pin_memory() if pinned else t

    ht, hl = host(tok), host(load)
    bad = off.copy()
    bad[n] = len(tok) + 1
    for o, rc_want in ((off, 0), (bad, pkg.SMETRIC_ERR_INVALID_ARG), (off, 0)):
        out = {k: host(np.full(n, 77, np.int32)) for k in ("instance", "local_hit", "global_hit")}
        out["session_key"] = host(np.full(n, 77, np.int64))
        rc = pkg.smetric_route_batch_host(ix.handle, ht, len(tok), host(o), n, hl, (1, 4, 2), out["instance"],
                                          out["local_hit"], out["global_hit"], out["session_key"])
        assert rc == rc_want
        for k, v in out.items():
            got = v.numpy().view(np.uint64) if k == "session_key" else v.numpy()
            if rc_want == 0:
                assert np.array_equal(got, want[k]), k
            else:
                assert np.all(v.numpy() == (-1 if k == "instance" else 0)), k
    assert ix.status() == 0
    ix.close()


@pytest.mark.parametrize("n", [3, 3000])
@pytest.mark.parametrize("side_stream", [False, True])
def test_pinned_inputs_are_read_in_stream_order(n, side_stream):
    """Loads, offsets and tokens that work enqueued before the call still writes."""
    rng = np.random.default_rng(n)
    N, B = 7, 2
    reqs = [rng.integers(0, 99, size=int(k), dtype=np.int32) for k in rng.integers(2, 9, size=n)]
    tok, off = pack(reqs)
    old = dict(tokens=rng.permutation(tok), offsets=np.minimum(off, off[n // 2]), load=np.arange(N, dtype=np.int64)[::-1].copy())
    new = dict(tokens=tok, offsets=off, load=np.arange(N, dtype=np.int64) * 1000)
    ix = make_index(N, B, 2, max_req=n, max_tok=len(tok), host_staging=True)
    want = gpu_route(ix, tok, off, new["load"], (1, 4, 2), want_hashes=False)
    stale = gpu_route(ix, old["tokens"], old["offsets"], old["load"], (1, 4, 2), want_hashes=False)
    assert not np.array_equal(want["instance"], stale["instance"])
    host = {k: torch.from_numpy(np.ascontiguousarray(v)).pin_memory() for k, v in old.items()}
    dev = {k: T(v) for k, v in new.items()}
    out = {k: torch.full((n,), 77, dtype=torch.int32).pin_memory() for k in ("instance", "local_hit", "global_hit")}
    out["session_key"] = torch.full((n,), 77, dtype=torch.int64).pin_memory()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if side_stream else torch.cuda.default_stream()):
        torch.cuda._sleep(40_000_000)  # some 20 ms
        for k in host:
            host[k].copy_(dev[k], non_blocking=True)
        rc = pkg.smetric_route_batch_host(ix.handle, host["tokens"], len(tok), host["offsets"], n, host["load"], (1, 4, 2),
                                          out["instance"], out["local_hit"], out["global_hit"], out["session_key"])
    assert rc == 0
    for k, v in out.items():
        assert np.array_equal(v.numpy().view(np.uint64) if k == "session_key" else v.numpy(), want[k]), k
    ix.close()
