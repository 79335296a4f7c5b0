"""Several indexes in one process: kernels that they share serve each of them,
whatever the others' block sizes and batch sizes are."""

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
