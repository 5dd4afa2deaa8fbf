"""The smallest orders of the local eigenproblem (Householder reduction and
bisection of T_i, orders 1 to 17 in one batch) and the batched solve on both
sides of the size from which its SpMV and prolongation take one warp a row for
all right-hand sides.

Bounds: the suite's 1e-8 on the eigenvalues, with 1e-10 absolute (T_i has norm
at most 1); one column of a batched one-level apply against the same column
alone, 1e-12 of its largest entry (FP64 sums of at most 8 terms in another
order are within 1e-15)."""
import numpy as np
import pytest

import synth
from oracle import amdd_oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _need():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")


def _mu(lam):
    with np.errstate(divide="ignore"):
        return np.sort(np.where(np.isinf(lam), 0.0, 1.0 / lam))


@pytest.mark.parametrize("tau", [0.5, 50.0])
def test_orders_1_to_17(tau):
    _need()
    from paper_2109_05908_gb300 import amdd as A
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    part = np.repeat(np.arange(17), np.arange(1, 18)).astype(np.int32)
    n = len(part)
    i = np.arange(n)
    d = 2.0 + 0.5 * np.sin(i)
    rows = np.concatenate([i, i[1:], i[:-1]])
    cols = np.concatenate([i, i[:-1], i[1:]])
    M = synth._csr_from_coo(n, rows, cols, np.concatenate([d + 0.6, -np.ones(2 * (n - 1))]))
    S = O.setup(M, part, 17, 1, tau)
    P = Preconditioner(DeviceMatrix(M), torch.from_numpy(part).cuda(), 17, 1, tau)
    try:
        for k, s in enumerate(S.subs):
            mo, mg = _mu(s.lam), _mu(A.get_eigenvalues(P.h, k))
            assert mo.shape == mg.shape and np.all(np.abs(mg - mo) <= 1e-8 * mo + 1e-10), k
    finally:
        P.close()


@pytest.mark.parametrize("m", [277, 279])  # 76729 and 77841 rows about the line at 77824
@pytest.mark.parametrize("nrhs", [2, 5, 8])
def test_batched_apply_columns(m, nrhs):
    _need()
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    M = synth.laplace2d(m)
    part = (np.arange(m * m) // 100).astype(np.int32)
    P = Preconditioner(DeviceMatrix(M), torch.from_numpy(part).cuda(), int(part[-1]) + 1, 1, 1e-17)
    try:
        b = torch.from_numpy(synth.rhs(M.n, 1, nrhs).reshape(nrhs, M.n)).cuda()
        z, one = torch.empty_like(b), torch.empty_like(b[0])
        P.apply(b, z, nrhs)
        x = torch.zeros_like(b)
        P.solve(b, x, nrhs, rtol=1e-8)
        for k in range(nrhs):
            P.apply(b[k].contiguous(), one)
            assert (z[k] - one).abs().max() <= 1e-12 * one.abs().max()
            r = synth.rhs(M.n, 1, nrhs).reshape(nrhs, M.n)[k] - _mul(M, x[k].cpu().numpy())
            assert np.linalg.norm(r) <= 1.5e-8 * np.linalg.norm(b[k].cpu().numpy())
    finally:
        P.close()


def _mul(M, x):
    return np.add.reduceat(M.val * x[M.colind], M.rowptr[:-1])
