"""The SpMV at its edges against a host product in FP64: row counts around a
block, values and columns that are not 16-byte aligned, rows far longer than
the average, empty rows, and the row lengths at which the lanes per row change.  The bar is len * u * sum |a x| per row (FP64 summation in any order)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _matrix(n, length, seed):
    rng = np.random.default_rng(seed)
    cnt = np.minimum(length(np.arange(n), rng), n).astype(np.int64)
    ptr = np.concatenate([[0], np.cumsum(cnt)])
    col = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in cnt] + [np.zeros(0, int)]).astype(np.int32)
    return ptr, col, rng.standard_normal(len(col)), rng.standard_normal(n)


SHAPES = {
    "1": (1, lambda r, g: np.ones(len(r))),
    "255_rows_of_0_to_9": (255, lambda r, g: g.integers(0, 10, len(r))),
    "257_rows_of_5": (257, lambda r, g: np.full(len(r), 5)),
    "1000_rows_of_7_or_8": (1000, lambda r, g: 7 + r % 2),
    "dense_block_among_short_rows": (2000, lambda r, g: np.where((r > 300) & (r < 420), 60, 2)),
    "512_rows_of_9": (512, lambda r, g: np.full(len(r), 9)),
    "512_rows_of_10": (512, lambda r, g: np.full(len(r), 10)),
    "513_rows_of_25": (513, lambda r, g: np.full(len(r), 25)),
    "300_rows_of_40_to_102": (300, lambda r, g: 40 + g.integers(0, 63, len(r))),
    "300_rows_of_128_to_260": (300, lambda r, g: 128 + g.integers(0, 133, len(r))),
    "400_rows_of_300": (400, lambda r, g: np.full(len(r), 300)),
}


@pytest.mark.parametrize("offset", (0, 1))
@pytest.mark.parametrize("name", SHAPES)
def test_spmv_forms(name, offset):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    n, length = SHAPES[name]
    ptr, col, val, x = _matrix(n, length, 3)
    nnz = len(col)
    dv = torch.zeros(nnz + 1, dtype=torch.float64, device="cuda")[offset:offset + nnz]
    dc = torch.zeros(nnz + 1, dtype=torch.int32, device="cuda")[offset:offset + nnz]
    dv.copy_(torch.from_numpy(val))
    dc.copy_(torch.from_numpy(col))
    dp, dx = torch.from_numpy(ptr).cuda(), torch.from_numpy(x).cuda()
    y = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    A.spmv(A.make_csr(n, nnz, dp.data_ptr(), dc.data_ptr(), dv.data_ptr()), dx.data_ptr(), y.data_ptr())
    row = np.repeat(np.arange(n), np.diff(ptr))
    ref, mag = np.zeros(n), np.zeros(n)
    np.add.at(ref, row, val * x[col])
    np.add.at(mag, row, np.abs(val * x[col]))
    assert (np.abs(y.cpu().numpy() - ref) <= 2 * (np.diff(ptr) + 1) * 2.0 ** -53 * mag).all()
