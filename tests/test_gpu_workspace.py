"""Workspace of the row sort per entry: 12 bytes of temporary keys and values where values are
8 bytes wide (8 where 4), and lists that stay well below one byte."""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_same, from_oracle

pytestmark = pytest.mark.gpu


class Counting:
    def __init__(self):
        from paper_2509_20776_gb300 import TorchAllocator
        self.inner, self.largest = TorchAllocator(0), 0

    def alloc(self, nbytes, stream):
        self.largest = max(self.largest, nbytes)
        return self.inner.alloc(nbytes, stream)

    def free(self, ptr, nbytes, stream):
        self.inner.free(ptr, nbytes, stream)


@pytest.mark.parametrize("vt", [np.float32, np.float64])
def test_permute_workspace_per_entry(vt):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2509_20776_gb300 import Context, build
    build.build()
    m, n, L = 1000, 1 << 16, 4200  # every row is cut into runs
    g = np.random.default_rng(1)
    col = np.concatenate([np.sort(g.choice(n, L, replace=False)) for _ in range(m)])
    O = oracle.CSR.of(m, n, np.arange(m + 1) * L, col, g.random(m * L).astype(vt))
    A = from_oracle(O)
    p, q = g.permutation(m).astype(np.int32), g.permutation(n).astype(np.int32)
    mem = Counting()
    ctx = Context(0, allocator=mem)
    try:
        B = ctx.sp_permute(A, torch.from_numpy(p).cuda(), torch.from_numpy(q).cuda())  # (outputs: PyTorch's)
        assert_same(B, oracle.permute(O, p, q), "permute")
    finally:
        ctx.close()
    nnz = m * L
    temp = nnz * (4 + np.dtype(vt).itemsize)
    maps = 64 * m + 8 * n  # row and column maps, bitmaps, row starts
    # the arena grows by a quarter more than was asked for
    assert mem.largest / 1.25 <= temp + maps + 0.6 * nnz
