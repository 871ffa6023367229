"""The row sort at the edges of its paths: tiles (windows that end inside a row, more rows
than fit one round, empty windows), single runs at every capacity, the key-range split,
skewed keys (a bucket of hundreds of keys is bucketed again), and a warp's short runs.
Results are moved, never computed, so they are compared bit for bit with the oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_same, from_oracle

pytestmark = pytest.mark.gpu

N = 1 << 20


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2509_20776_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


def matrix(lens, skew, vt, seed):
    """Rows of the given lengths; skew: a row's columns crowd at the top of the range."""
    g = np.random.default_rng(seed)
    cols = []
    for L in lens:
        if skew and L > 1:
            c = np.concatenate([[0], N - 1 - np.arange(L - 1)[::-1] * (1 + L % 3)])
        else:
            c = np.sort(g.choice(N, L, replace=False))
        cols.append(c)
    col = np.concatenate(cols) if cols else np.zeros(0, np.int64)
    rp = np.concatenate([[0], np.cumsum(lens)])
    return oracle.CSR.of(len(lens), N, rp, col.astype(np.int64), g.random(len(col)).astype(vt))


EDGES = [0, 1, 2, 31, 32, 33, 127, 128, 129, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 4095, 4096, 4097, 8192]
MIXES = {
    "edges": EDGES * 2,
    "rounds": [512, 511, 400, 500, 300, 512, 512, 3, 0, 512, 200, 509] * 20,  # windows of more than a round
    "tiny": [3, 0, 1, 2, 5, 0, 0, 1] * 700,
    "windows": [5, 4000, 0, 0, 7, 9000, 1, 0, 70000, 2],  # empty windows inside longer rows
    "single": [1],
}


@pytest.mark.parametrize("vt", [np.float32, np.float64])
@pytest.mark.parametrize("ci", [torch.int32, torch.int64])
@pytest.mark.parametrize("mix", sorted(MIXES))
@pytest.mark.parametrize("tile_shape", [0, 1])
def test_permute_row_lengths(ctx, mix, tile_shape, ci, vt):
    A = matrix(MIXES[mix], False, vt, 1)
    g = np.random.default_rng(2)
    p, q = g.permutation(A.nrows).astype(np.int32), g.permutation(N).astype(np.int32)
    ctx.set_shapes(tile_shape=tile_shape)
    try:
        B = ctx.sp_permute(from_oracle(A, colidx_dtype=ci), torch.from_numpy(p).cuda(), torch.from_numpy(q).cuda())
    finally:
        ctx.set_shapes(tile_shape=-1)
    assert_same(B, oracle.permute(A, p, q), mix)


@pytest.mark.parametrize("heavy", [128, 512])
@pytest.mark.parametrize("skew", [False, True])
@pytest.mark.parametrize("mix", ["edges", "rounds", "windows"])
def test_sort_rows_in_place(ctx, mix, skew, heavy):
    A = matrix(MIXES[mix], skew, np.float32, 3)
    g = np.random.default_rng(4)
    M = from_oracle(A)
    order = np.concatenate([b + g.permutation(e - b) for b, e in zip(A.rowptr[:-1], A.rowptr[1:])])
    order = torch.from_numpy(order).cuda()
    M.colidx, M.values = M.colidx[order].contiguous(), M.values[order].contiguous()
    ctx.set_shapes(heavy=heavy)
    try:
        ctx.sp_sort_rows(M)
    finally:
        ctx.set_shapes(heavy=-1)
    assert_same(M, A, f"{mix} {skew}")


@pytest.mark.parametrize("nj", [40, 300, N // 8, N // 2])
def test_extract_queues_short_runs(ctx, nj):
    """Rows of 65 to 1024 source entries whose kept part has a few to some hundred entries,
    and longer ones whose key-range split leaves short groups."""
    A = matrix([65, 66, 96, 128, 129, 200, 256, 257, 400, 512, 700, 1000, 1024] * 5 +
               list(range(8200, 30000, 700)), False, np.float32, 5)
    g = np.random.default_rng(6)
    I, J = g.permutation(A.nrows).astype(np.int32), g.permutation(N)[:nj].astype(np.int32)
    B = ctx.sp_extract(from_oracle(A), torch.from_numpy(I).cuda(), torch.from_numpy(J).cuda())
    assert_same(B, oracle.extract(A, I, J), f"{nj}")


def test_repeated_row_in_p_stays_inside(ctx):
    """p repeats the longest row: reported, and no write leaves the output arrays."""
    from paper_2509_20776_gb300 import CSR, SpError
    A = from_oracle(matrix([4000, 3, 600, 2, 0, 100], False, np.float32, 7))
    p = torch.zeros(6, dtype=torch.int32, device="cuda")
    q = torch.randperm(N, device="cuda").to(torch.int32)
    pad = 20000
    col = torch.full((A.nnz + pad,), 7, dtype=torch.int32, device="cuda")
    val = torch.full((A.nnz + pad,), 7.0, device="cuda")
    out = CSR(6, N, torch.empty(7, dtype=torch.int64, device="cuda"), col[:A.nnz], val[:A.nnz])
    with pytest.raises(SpError) as e:
        ctx.sp_permute(A, p, q, out=out)
    assert e.value.name == "SP_ERR_NOT_PERMUTATION"
    assert bool((col[A.nnz:] == 7).all()) and bool((val[A.nnz:] == 7.0).all())


LARGE = EDGES * 5  # more entries than one launch for all runs takes: each run by the kernel of its length


@pytest.mark.parametrize("vt", [np.float32, np.float64])
@pytest.mark.parametrize("skew", [False, True])  # (the identity keeps the columns crowded: heavy buckets)
@pytest.mark.parametrize("tile_shape", [0, 1])
def test_permute_runs_by_length(ctx, tile_shape, skew, vt):
    assert sum(LARGE) > 1 << 17
    A = matrix(LARGE, skew, vt, 8)
    g = np.random.default_rng(9)
    p = g.permutation(A.nrows).astype(np.int32)
    q = (np.arange(N) if skew else g.permutation(N)).astype(np.int32)
    ctx.set_shapes(tile_shape=tile_shape)
    try:
        B = ctx.sp_permute(from_oracle(A), torch.from_numpy(p).cuda(), torch.from_numpy(q).cuda())
    finally:
        ctx.set_shapes(tile_shape=-1)
    assert_same(B, oracle.permute(A, p, q), f"{tile_shape} {skew}")


@pytest.mark.parametrize("vt", [np.float32, np.float64])
@pytest.mark.parametrize("skew", [False, True])
@pytest.mark.parametrize("tile_shape", [0, 1])
def test_sort_runs_in_place_by_length(ctx, tile_shape, skew, vt):
    A = matrix(LARGE, skew, vt, 10)
    g = np.random.default_rng(11)
    M = from_oracle(A)
    order = np.concatenate([b + g.permutation(e - b) for b, e in zip(A.rowptr[:-1], A.rowptr[1:])])
    order = torch.from_numpy(order).cuda()
    M.colidx, M.values = M.colidx[order].contiguous(), M.values[order].contiguous()
    ctx.set_shapes(tile_shape=tile_shape)
    try:
        ctx.sp_sort_rows(M)
    finally:
        ctx.set_shapes(tile_shape=-1)
    assert_same(M, A, f"{tile_shape} {skew}")
