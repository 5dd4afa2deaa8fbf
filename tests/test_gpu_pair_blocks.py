"""The block-pair Jacobi on the tensor cores at the edges of its blocks: orders
that fill the last 32-row block, leave one row in it, or need an empty one, and
leading dimensions off the 16-byte boundary (FP64: the FP32 stage of [X | I]).

FP64 setup: singular values to the suite's 1e-10 of sigma_1.  Mixed setup: the same selection and PCG count (one more or less) as
the FP64 one."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,rows", [(32, 31), (41, 24), (33, 31), (41, 25)])
def test_block_edges(m, rows):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    M = synth.laplace2d(m)
    part = (np.arange(m * m) // m >= rows).astype(np.int32)
    D = np.zeros((m * m, m * m))
    rp, ci = np.asarray(M.rowptr), np.asarray(M.colind)
    D[np.repeat(np.arange(m * m), np.diff(rp)), ci] = np.asarray(M.val)
    dM, dp = DeviceMatrix(M), torch.from_numpy(part).cuda()
    b = torch.from_numpy(synth.rhs(M.n, 0)).cuda()
    out = []
    for precision in (0, 1):
        o = A.opts_default()
        o.precision = precision
        P = Preconditioner(dM, dp, 2, 1, 50.0, o)
        try:
            info = P.info()
            assert info.pair_stats[1] > 0  # the block-pair form ran
            x = torch.zeros_like(b)
            st = P.solve(b, x, rtol=1e-8)
            assert st.converged == 1 and st.true_rel_residual <= 2e-8
            out.append((info.n_C, st.iterations))
            if precision == 0:
                for i in range(2):
                    so = np.linalg.svd(D[np.abs(D[:, part == i]).sum(1) > 0], compute_uv=False)
                    sg = np.sort(np.asarray(A.get_singular_values(P.h, i)))[::-1]
                    assert sg.shape == so.shape and np.abs(sg - so).max() <= 1e-10 * so[0]
        finally:
            P.close()
    assert out[0][0] == out[1][0] and abs(out[0][1] - out[1][1]) <= 1
