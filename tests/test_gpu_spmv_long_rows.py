"""The SpMV where the lanes per row and the treatment of long rows change: row
counts on both sides of the thread limit that doubles the lanes, and rows at,
just above and far above the length from which a whole warp takes a row (the
larger of 64 and four times the average), first, last and neighbouring rows of
a warp among them.  Bar as for the other forms: len * u * sum |a x| per row,
FP64 summation in any order.  The residual form and the form with the fused dot
product run through GMRES and PCG on an arrow matrix."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# rows, their length, lengths of some rows
SHAPES = {
    "2000_of_9": (2000, 9, {}),
    "2001_of_32": (2001, 32, {}),
    "4000_of_64": (4000, 64, {}),
    "4001_of_64": (4001, 64, {}),
    "64001_of_5_rows_of_64_65_66": (64001, 5, {0: 64, 1: 65, 2: 66, 31: 65, 32: 5000, 64000: 65}),
    "70000_of_12_neighbours": (70000, 12, {k: 70 + k for k in range(40)}),
    "40000_of_30_rows_of_120_to_122": (40000, 30, {7: 120, 8: 121, 9: 122, 39999: 3000, 15: 0}),
    "500_of_20_one_full": (500, 20, {499: 500}),
}


@pytest.mark.parametrize("name", SHAPES)
def test_spmv_long_rows(name):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    n, length, some = SHAPES[name]
    rng = np.random.default_rng(5)
    cnt = np.full(n, length)
    for r, c in some.items():
        cnt[r] = c
    ptr = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int64)
    row = np.repeat(np.arange(n), cnt)
    col = ((row + 3 * (np.arange(len(row)) - ptr[row])) % n).astype(np.int32)
    val, x = rng.standard_normal(len(row)), rng.standard_normal(n)
    dev = [torch.from_numpy(v).cuda() for v in (ptr, col, val, x)]
    y = torch.full((n,), 7.0, dtype=torch.float64, device="cuda")
    A.spmv(A.make_csr(n, len(row), *(t.data_ptr() for t in dev[:3])), dev[3].data_ptr(), y.data_ptr())
    ref, mag = np.zeros(n), np.zeros(n)
    np.add.at(ref, row, val * x[col])
    np.add.at(mag, row, np.abs(val * x[col]))
    assert (np.abs(y.cpu().numpy() - ref) <= 2 * (cnt + 1) * 2.0 ** -53 * mag).all()


def test_solves_with_a_long_row():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    n = 600
    i = np.arange(n)
    hub, rest = np.zeros(n - 1, int), i[1:]
    M = synth._csr_from_coo(n, np.concatenate([i, hub, rest, i[1:], i[:-1]]), np.concatenate([i, rest, hub, i[:-1], i[1:]]),
                            np.concatenate([np.where(i == 0, float(n), 5.0), np.full(2 * (n - 1), -0.5), -np.ones(2 * (n - 1))]))
    D = np.zeros((n, n))
    D[np.repeat(i, np.diff(M.rowptr)), M.colind] = M.val
    part = (i * 4 // n).astype(np.int32)
    P = Preconditioner(DeviceMatrix(M), torch.from_numpy(part).cuda(), 4, 1, 0.5)
    try:
        b = synth.rhs(n, 0)
        bd = torch.from_numpy(b).cuda()
        for solve in (P.solve, P.gmres):
            x = torch.zeros_like(bd)
            st = solve(bd, x, rtol=1e-8)
            assert st.converged == 1
            assert np.linalg.norm(b - D @ x.cpu().numpy()) <= 1.5e-8 * np.linalg.norm(b)
            assert st.true_rel_residual <= 1.5e-8
    finally:
        P.close()
