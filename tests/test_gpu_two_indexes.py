"""Several indexes in one process: kernels that they share serve each of them,
whatever the others' block sizes and batch sizes are."""

import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import paper_2607_08565_gb300 as pkg
from gpu_util import T, gpu_hashes, make_index
from synth.traces import pack

pytestmark = pytest.mark.gpu


def _noalloc(tok, off, B):
    n, nb = len(off) - 1, len(tok) // B
    h, sk = torch.zeros(max(nb, 1), dtype=torch.int64, device="cuda"), torch.zeros(n, dtype=torch.int64, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    rc = pkg.smetric_block_hashes_noalloc(T(tok), len(tok), T(off), n, B, 2, 0, sk, h, nb, status)
    assert rc == 0 and int(status.item()) == 0
    return h.cpu().numpy().view(np.uint64)[:int((np.diff(off) // B).sum())]


@pytest.mark.parametrize("large,small", [(256, 20), (250, 2), (128, 16), (32, 12)])
def test_block_sizes_in_turn(large, small):
    rng = np.random.default_rng(large)
    reqs = [rng.integers(0, 151936, size=int(k), dtype=np.int32) for k in rng.integers(0, 9 * large, size=55)]
    tok, off = pack(reqs)
    want = {B: np.concatenate([oracle.block_hashes(r, B) for r in reqs]) for B in (large, small)}
    first, second = (make_index(3, B, 2, max_tok=len(tok)) for B in (large, small))
    for ix, B in ((first, large), (second, small), (first, large), (None, small), (first, large), (None, large), (second, small)):
        got = gpu_hashes(ix, tok, off)[0] if ix else _noalloc(tok, off, B)
        assert np.array_equal(got, want[B]), B
    first.close()
    second.close()


@pytest.mark.parametrize("commit,shapes", [(False, ((7, 2000), (7, 6080))), (True, ((190, 5), (256, 5)))])
def test_threads_on_indexes_of_their_own(commit, shapes):
    """Eight threads, each with an index and a stream; their batches want different amounts of shared memory."""
    B, rounds, L = 2, 5000, pkg.lib()
    failed = []

    def work(N, n):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            ix = make_index(N, B, 1, max_req=n, max_tok=n * B)
            off = T(np.arange(n + 1, dtype=np.int64) * B)
            tok, load, out = T(np.zeros(n * B, np.int32)), T(np.zeros(N, np.int64)), T(np.zeros((3, n), np.int32))
            h = T(np.arange(2, n + 2))
            if commit:
                ix.set_lru(8)
            a, s, w = out.data_ptr(), stream.cuda_stream, pkg.smetric_weights(1, 4, 2)
            stream.synchronize()
            for i in range(rounds):
                if commit:
                    rc = L.smetric_index_commit_batch(ix.handle, off.data_ptr(), n, a, a + 4 * n, h.data_ptr(), 0, None, s)
                else:
                    rc = L.smetric_route_batch(ix.handle, tok.data_ptr(), n * B, off.data_ptr(), n, load.data_ptr(), w,
                                               a, a + 4 * n, a + 8 * n, h.data_ptr(), None, 0, s)
                failed.extend([rc] if rc else [])
                if i % 200 == 0:
                    stream.synchronize()
            ix.check()
            done.append(n)

    done = []
    threads = [threading.Thread(target=work, args=shapes[k % 2]) for k in range(8)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed and len(done) == 8
