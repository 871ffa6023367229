"""A row pointer that does not ascend: a scan that gives up waiting (SP_ERR_TIMEOUT) leaves one
behind for the kernels launched after it, and a caller's own may hold anything.  Each call
reports its error, writes nothing outside its output arrays, and leaves the context usable."""
import ctypes
from contextlib import contextmanager

import numpy as np
import pytest
import torch

import oracle
from helpers import assert_same, from_oracle

pytestmark = pytest.mark.gpu

N = 1 << 20
PAD = 1 << 16


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2509_20776_gb300 import Context, build
    build.build()
    c = Context(0)
    yield c
    c.close()


@contextmanager
def held(ctx):
    """Tile 1 of every scan never publishes: the row pointer drops to 0 where tile 2 begins
    (row 2048 of a scan of at most 2^17 rows)."""
    from paper_2509_20776_gb300 import SP_OPT_SCAN_HOLD_TILE, SP_OPT_SPIN_LIMIT
    ctx.set_option(SP_OPT_SPIN_LIMIT, 2000)
    ctx.set_option(SP_OPT_SCAN_HOLD_TILE, 1)
    try:
        yield
    finally:
        ctx.set_option(SP_OPT_SCAN_HOLD_TILE, -1)
        ctx.set_option(SP_OPT_SPIN_LIMIT, -1)


def matrix(lens, seed, n=N):
    g = np.random.default_rng(seed)
    lens = np.asarray(lens)
    col = np.concatenate([np.sort(g.choice(n, int(x), replace=False)) for x in lens])
    return oracle.CSR.of(len(lens), n, np.concatenate([[0], np.cumsum(lens)]), col, g.random(len(col)).astype(np.float32))


class Padded:
    """Output arrays with PAD words before and after that nothing may write."""

    def __init__(self, nrows, ncols, nnz, vt=torch.float32):
        from paper_2509_20776_gb300 import CSR
        self.col = torch.full((nnz + 2 * PAD,), 7, dtype=torch.int32, device="cuda")
        self.val = torch.full((nnz + 2 * PAD,), 7.0, dtype=vt, device="cuda")
        self.out = CSR(nrows, ncols, torch.empty(nrows + 1, dtype=torch.int64, device="cuda"),
                       self.col[PAD:PAD + nnz], self.val[PAD:PAD + nnz])

    def check(self):
        for a in (self.col, self.val):
            assert bool((a[:PAD] == 7).all()) and bool((a[-PAD:] == 7).all())


KINDS = {  # row lengths of a matrix of 6000 rows
    "sparse": lambda g: g.integers(0, 4, 6000),       # the drop lies inside a window
    "tiles": lambda g: g.integers(0, 513, 6000),
    "runs": lambda g: np.where(g.random(6000) < 0.1, g.integers(513, 2500, 6000), g.integers(0, 30, 6000)),
    "long": lambda g: np.where(g.random(6000) < 0.03, g.integers(4097, 20000, 6000), g.integers(0, 9, 6000)),
}


def expect(ctx, name, call):
    from paper_2509_20776_gb300 import SpError
    with pytest.raises(SpError) as e:
        call()
        ctx.sync()
    assert e.value.name == name


def idx(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randperm(n, generator=g, device="cuda").to(torch.int32)


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("tile_shape,n", [(0, N), (1, N), (0, 1 << 24)])  # (keys of 24 bits: the fine split follows)
@pytest.mark.parametrize("columns", [True, False])  # (rows alone: gathered without a sort)
def test_permute(ctx, kind, tile_shape, n, columns):
    O = matrix(KINDS[kind](np.random.default_rng(1)), 2, n)
    A, p, q = from_oracle(O), idx(6000, 3), idx(n, 4) if columns else None
    P = Padded(6000, n, A.nnz)
    ctx.set_shapes(tile_shape=tile_shape)
    try:
        with held(ctx):
            expect(ctx, "SP_ERR_TIMEOUT", lambda: ctx.sp_permute(A, p, q, out=P.out))
        P.check()
        assert_same(ctx.sp_permute(A, p, q), oracle.permute(O, p.cpu().numpy(), q.cpu().numpy() if columns else None), kind)
    finally:
        ctx.set_shapes(tile_shape=-1)


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("columns", [True, False])
def test_permute_batch(ctx, kind, columns):
    mats = [from_oracle(matrix(KINDS[kind](np.random.default_rng(s))[:2500], s)) for s in (5, 6, 7)]
    reqs = [(k, idx(2500, 10 + k), idx(N, 20 + k) if columns else None) for k in range(3)]
    bt = ctx.permute_batch(mats, reqs)
    try:
        P = Padded(7500, N, sum(m.nnz for m in mats))
        with held(ctx):
            expect(ctx, "SP_ERR_TIMEOUT", lambda: bt.fill(P.out))
        P.check()
    finally:
        bt.close()


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("identify", [0, 1])
def test_extract_batch_run(ctx, kind, identify):
    """A run counts again: its row pointer and (identify 0) its ranks come from scans."""
    mats = [from_oracle(matrix(KINDS[kind](np.random.default_rng(s))[:3000], s)) for s in (18, 19)]
    reqs = [(k % 2, idx(3000, 40 + k), idx(N, 50 + k)[:N // 2].contiguous()) for k in range(4)]
    ctx.set_shapes(identify=identify)
    try:
        bt = ctx.extract_batch(mats, reqs)
        try:
            P = Padded(12000, N, bt.nnz)
            with held(ctx):
                expect(ctx, "SP_ERR_TIMEOUT", lambda: bt.run(P.out))
            P.check()
        finally:
            bt.close()
    finally:
        ctx.set_shapes(identify=-1)


def assign_plan(ctx, A, I, J, B, mode=0):
    plan, nnz = ctypes.c_void_p(), ctypes.c_int64()
    st = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    ctx._check(ctx.lib.sp_assign_count(ctx.handle, ctypes.byref(A.desc()), ctypes.c_void_p(I.data_ptr()), I.numel(),
                                       ctypes.c_void_p(J.data_ptr()), J.numel(), 0, ctypes.byref(B.desc()), mode,
                                       ctypes.byref(plan), ctypes.byref(nnz), st), "sp_assign_count")
    return plan, nnz.value, st


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_assign_permute(ctx, kind):
    A = from_oracle(matrix(KINDS[kind](np.random.default_rng(8)), 9))
    I, J = idx(6000, 30)[:900].contiguous(), idx(N, 31)[:3000].contiguous()
    B = from_oracle(matrix(np.random.default_rng(10).integers(0, 9, 900), 11, 3000))
    p, q = idx(6000, 32), idx(N, 33)
    plan, nnz, st = assign_plan(ctx, A, I, J, B)
    try:
        P = Padded(6000, N, nnz)
        d = P.out.desc()
        with held(ctx):
            expect(ctx, "SP_ERR_TIMEOUT", lambda: ctx._check(ctx.lib.sp_assign_permute_fill(
                ctx.handle, plan, ctypes.c_void_p(p.data_ptr()), ctypes.c_void_p(q.data_ptr()), ctypes.byref(d), st), ""))
        P.check()
    finally:
        ctx.lib.sp_plan_destroy(ctx.handle, plan)


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("fault", ["drop", "negative", "past", "comb"])
def test_sort_rows_of_a_bad_row_pointer(ctx, kind, fault):
    O = matrix(KINDS[kind](np.random.default_rng(12)), 13)
    rp = O.rowptr.copy()
    if fault == "drop":
        rp[3000:] -= rp[3000]
    elif fault == "negative":
        rp[100] = -(1 << 40)
    elif fault == "past":
        rp[2000] = rp[-1] + 12345
    else:  # every second row lies on all the later ones: more long rows than the entries can hold
        rp[1::2] = rp[-1]
    P = Padded(len(rp) - 1, N, len(O.colidx))
    P.out.rowptr = torch.from_numpy(rp).cuda()
    P.out.colidx.copy_(torch.from_numpy(O.colidx.astype(np.int32)))
    expect(ctx, "SP_ERR_NOT_CANONICAL", lambda: ctx.sp_sort_rows(P.out))
    P.check()


@pytest.mark.parametrize("mode", [0, 1])  # REPLACE: merged beside the copy; SELECT2ND: staged
@pytest.mark.parametrize("runs", [1, 5])  # of rows of I: segments of one row, of some rows
def test_assign(ctx, mode, runs):
    """The segments' scan takes 32 rows a value, tiles of 1024: the timeout needs 2^16 rows."""
    m = 200_000
    g = np.random.default_rng(14)
    O = matrix(g.integers(0, 5, m), 15, 5000)
    A = from_oracle(O)
    r = np.arange(m)
    rows = r[(r // runs) % 2 == 0].astype(np.int32)
    I, J = torch.from_numpy(rows).cuda(), idx(5000, 34)[:300].contiguous()
    Bo = matrix(g.integers(0, 4, len(rows)), 16, 300)
    B = from_oracle(Bo)
    plan, nnz, st = assign_plan(ctx, A, I, J, B, mode)
    try:
        P = Padded(m, 5000, nnz)
        d = P.out.desc()
        with held(ctx):
            expect(ctx, "SP_ERR_TIMEOUT", lambda: ctx._check(ctx.lib.sp_assign_fill(ctx.handle, plan, ctypes.byref(d), st), ""))
        P.check()
    finally:
        ctx.lib.sp_plan_destroy(ctx.handle, plan)
    assert_same(ctx.sp_assign(A, I, J, B, mode=mode), oracle.assign(O, rows, J.cpu().numpy(), Bo, mode), f"{mode} {runs}")


@pytest.mark.parametrize("kind", sorted(KINDS))
def test_sort_rows_of_a_slice(ctx, kind):
    """Rows of a larger matrix: a row pointer that starts above 0 and ends below the entries."""
    from paper_2509_20776_gb300 import CSR
    O = matrix(KINDS[kind](np.random.default_rng(16)), 17)
    g = np.random.default_rng(18)
    r0, r1 = 2500, 4700
    lo, hi = int(O.rowptr[r0]), int(O.rowptr[r1])
    assert lo > 2048 and hi < len(O.colidx)  # beyond the first window
    col, val = O.colidx.copy(), O.values.copy()
    for b, e in zip(O.rowptr[r0:r1], O.rowptr[r0 + 1:r1 + 1]):
        o = b + g.permutation(e - b)
        col[b:e], val[b:e] = O.colidx[o], O.values[o]
    M = CSR(r1 - r0, N, torch.from_numpy(O.rowptr[r0:r1 + 1]).cuda(), torch.from_numpy(col.astype(np.int32)).cuda(),
            torch.from_numpy(val).cuda())
    ctx.sp_sort_rows(M)
    assert np.array_equal(M.colidx.cpu().numpy(), O.colidx)
    assert np.array_equal(M.values.cpu().numpy(), O.values)
