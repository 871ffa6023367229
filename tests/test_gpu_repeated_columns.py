"""Columns that repeat within a row longer than one run (no canonical matrix has them): the
key-range split cannot part equal keys, so it reports the row, whatever the width of the keys."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ncols", [3000, 1 << 20, 1 << 22, (1 << 22) + 1, 1 << 26])
def test_sort_rows_reports_them(ncols):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2509_20776_gb300 import CSR, Context, SpError, build
    build.build()
    ctx = Context(0)
    try:
        L = 6000  # entries, all with the same column
        M = CSR(2, ncols, torch.tensor([0, L, L + 3], device="cuda"),
                torch.cat([torch.full((L,), 7), torch.tensor([2, 1, 0])]).to(device="cuda", dtype=torch.int32),
                torch.rand(L + 3, device="cuda"))
        with pytest.raises(SpError) as e:
            ctx.sp_sort_rows(M)
        assert e.value.name == "SP_ERR_INTERNAL"
        assert M.colidx[L:].tolist() == [0, 1, 2]
    finally:
        ctx.close()
