"""The extraction's count and fill at the edges of their paths: rows around the lane path's and
the warp paths' lengths, at every alignment of a row's first entry, near both ends of the
arrays (where a lane loads entry by entry), all index and value widths, general and
ascending J, single calls and a batch.  Compared bit for bit with the oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_same, from_oracle

pytestmark = pytest.mark.gpu

N = 5000


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2509_20776_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


def matrix(lens, vt, seed):
    g = np.random.default_rng(seed)
    col = np.concatenate([np.sort(g.choice(N, L, replace=False)) for L in lens])
    return oracle.CSR.of(len(lens), N, np.concatenate([[0], np.cumsum(lens)]), col, g.random(len(col)).astype(vt))


LENS = [1, 2, 0, 3, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 4, 6, 1]
SHAPES = {"edges": LENS * 4, "one": [1], "two": [2, 1], "mesh": [5, 4, 5, 3] * 100, "tail": [40, 8, 8, 1]}


@pytest.mark.parametrize("vt", [np.float32, np.float64])
@pytest.mark.parametrize("ci", [torch.int32, torch.int64])
@pytest.mark.parametrize("ascending", [False, True])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_extract_row_lengths(ctx, shape, ascending, ci, vt):
    A = matrix(SHAPES[shape], vt, 1)
    g = np.random.default_rng(2)
    I = np.concatenate([np.arange(A.nrows), g.integers(0, A.nrows, 40)]).astype(np.int32)
    dA = from_oracle(A, colidx_dtype=ci)
    for k in (1, N // 9, N // 2, N):
        J = g.permutation(N)[:k].astype(np.int32)
        J = np.sort(J) if ascending else J
        if k == N:  # (consecutive when ascending: leave one out)
            J = J[J != 7]
        B = ctx.sp_extract(dA, torch.from_numpy(I).cuda(), torch.from_numpy(J).cuda())
        assert_same(B, oracle.extract(A, I, J), f"{shape} {k}")


@pytest.mark.parametrize("vt", [np.float32, np.float64])
def test_batch_row_lengths(ctx, vt):
    g = np.random.default_rng(3)
    mats = [matrix(SHAPES[k], vt, 4 + i) for i, k in enumerate(sorted(SHAPES))]
    reqs = []
    for k in range(60):
        A = mats[k % len(mats)]
        reqs.append((k % len(mats), g.integers(0, A.nrows, int(g.integers(1, 90))).astype(np.int32),
                     g.permutation(N)[:int(g.integers(1, N))].astype(np.int32)))
    out, first = ctx.sp_extract_batch([from_oracle(A) for A in mats],
                                      [(m, torch.from_numpy(I).cuda(), torch.from_numpy(J).cuda()) for m, I, J in reqs])
    rp, col, val = out.rowptr.cpu().numpy(), out.colidx.cpu().numpy(), out.values.cpu().numpy()
    for k, (m, I, J) in enumerate(reqs):
        want = oracle.extract(mats[m], I, J)
        r0, r1 = first[k], first[k + 1]
        assert np.array_equal(rp[r0:r1 + 1] - rp[r0], want.rowptr), k
        assert np.array_equal(col[rp[r0]:rp[r1]], want.colidx), k
        assert np.array_equal(val[rp[r0]:rp[r1]], want.values), k
