"""The assignment's copy and merge at the edges of their paths: chunks with more segments than
a warp holds, runs of rows of I (one segment in place of many), rows longer than a chunk,
empty rows at both ends, all widths; merged in place (REPLACE) and staged (union modes).
Compared bit for bit with the oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_same, from_oracle

pytestmark = pytest.mark.gpu

N = 6000


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2509_20776_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


def matrix(lens, ncols, vt, g):
    col = np.concatenate([np.sort(g.choice(ncols, L, replace=False)) for L in lens] or [np.zeros(0, np.int64)])
    return oracle.CSR.of(len(lens), ncols, np.concatenate([[0], np.cumsum(lens)]), col, g.random(len(col)).astype(vt))


SHAPES = {
    "short": [0, 1, 2, 3, 1, 0, 2] * 300,
    "mixed": [0, 33, 5000, 1, 64, 0, 2047, 2048, 2049, 7, 31, 32] * 4,
    "one": [5],
    "ends": [0, 0, 0, 40, 1500, 3, 0, 0],
}


def rows_of(kind, m, g):
    if kind == "alternate":
        return np.arange(0, m, 2)
    if kind == "runs":
        r = np.arange(m)
        return r[(r // 37) % 2 == 0]
    if kind == "all":
        return np.arange(m)
    if kind == "none":
        return np.zeros(0, np.int64)
    return g.permutation(m)[:max(1, m // 5)]


@pytest.mark.parametrize("vt,ci", [(np.float32, torch.int32), (np.float64, torch.int32), (np.float32, torch.int64),
                                   (np.float64, torch.int64)])
@pytest.mark.parametrize("mode", ["replace", "second"])
@pytest.mark.parametrize("kind", ["alternate", "runs", "all", "none", "random"])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_assign_segments(ctx, shape, kind, mode, vt, ci):
    from paper_2509_20776_gb300 import _binding as b
    g = np.random.default_rng(len(shape) * 7 + len(kind))
    A = matrix(SHAPES[shape], N, vt, g)
    I = rows_of(kind, A.nrows, g).astype(np.int32)
    J = g.permutation(N)[:400].astype(np.int32)
    B = matrix(g.integers(0, 33, len(I)), len(J), vt, g)
    if len(I) == 0:
        B = oracle.CSR.of(0, len(J), [0], np.zeros(0, np.int64), np.zeros(0, vt))
    want = oracle.assign(A, I, J, B) if mode == "replace" else oracle.assign(A, I, J, B, 1)
    got = ctx.sp_assign(from_oracle(A, colidx_dtype=ci), torch.from_numpy(I).cuda(), torch.from_numpy(J).cuda(),
                        from_oracle(B, colidx_dtype=ci),
                        mode=b.SP_ASSIGN_REPLACE if mode == "replace" else b.SP_ASSIGN_SELECT2ND)
    assert_same(got, want, f"{shape} {kind} {mode}")
