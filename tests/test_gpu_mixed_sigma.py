"""Singular values of the X_i in the mixed form from the block-pair Jacobi, on the tensor
cores and without, against the FP64 SVD, at orders that fill the last 32-row block,
leave one row in it, or need an empty one, with one inner sweep per visit and several.

Bar, relative to the largest singular value.  A row is rewritten once per visit of its
block, V = sweeps * (blocks - 1) visits.  The tensor core adds the 64 products in
eight steps and truncates each sum, so a visit shortens a row by at most 8 * 2^-23; the
7 rounds per inner sweep that build the rotation add 31 rounding errors each, of either
sign; and rows count as orthogonal at 8 sqrt(columns) 2^-23:
(8 V + sqrt(V * 7 * 31 * inner) + 8 sqrt(columns)) * 2^-23."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("inner", [1, 3])
@pytest.mark.parametrize("tensor_cores", [1, 0])
@pytest.mark.parametrize("m,rows", [(32, 31), (41, 24), (33, 31), (41, 25)])
def test_mixed_singular_values(m, rows, tensor_cores, inner):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    M = synth.laplace2d(m)
    part = (np.arange(m * m) // m >= rows).astype(np.int32)
    D = np.zeros((m * m, m * m))
    D[np.repeat(np.arange(m * m), np.diff(M.rowptr)), M.colind] = M.val
    o = A.opts_default()
    o.precision, o.tensor_cores, o.jacobi_inner_sweeps = 1, tensor_cores, inner
    P = Preconditioner(DeviceMatrix(M), torch.from_numpy(part).cuda(), 2, 1, 50.0, o)
    try:
        info = P.info()
        assert info.pair_stats[1] > 0  # the block-pair form ran
        worst = []
        for i in range(2):
            X = D[np.abs(D[:, part == i]).sum(1) > 0]
            X = X[:, np.abs(X).sum(0) > 0]
            so = np.linalg.svd(X, compute_uv=False)
            sg = np.sort(np.asarray(A.get_singular_values(P.h, i)))[::-1]
            assert sg.shape == so.shape
            blocks = max(2, 2 * -(-X.shape[0] // 64))
            V = info.sweeps_svd * (blocks - 1)
            bar = (8 * V + np.sqrt(V * 7 * 31 * inner) + 8 * np.sqrt(X.shape[1])) * 2.0 ** -23
            worst.append((np.abs(sg - so).max() / so[0], bar))
            print(f"\n[sigma] {X.shape} tc {tensor_cores} inner {inner} sweeps {info.sweeps_svd}: "
                  f"{worst[-1][0]:.2e} (bar {bar:.2e}, mean {np.mean(sg - so) / so[0]:.1e})")
        assert all(w <= b for w, b in worst), worst
    finally:
        P.close()
