"""The prolongation of several right-hand sides beyond the lines at which one
thread takes an unknown for all of them: 77,824 unknowns for two or three vectors,
311,296 for more.  One column of a batched one-level apply against the same column
alone, 1e-12 of its largest entry (FP64 sums of at most 8 terms in another order
are within 1e-15), and batched solves, whose dot products come from the same
kernel, to the true residual."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("m,nrhs", [(279, 3), (279, 4), (557, 4), (559, 4), (559, 8)])
def test_batched_lines(m, nrhs):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    M = synth.laplace2d(m)
    M.val[M.val > 0] = 4.5  # a few iterations
    part = (np.arange(m * m) // 100).astype(np.int32)
    P = Preconditioner(DeviceMatrix(M), torch.from_numpy(part).cuda(), int(part[-1]) + 1, 1, 1e-17)
    try:
        b = synth.rhs(M.n, 1, nrhs).reshape(nrhs, M.n)
        bd = torch.from_numpy(b).cuda()
        z, one, x = torch.empty_like(bd), torch.empty_like(bd[0]), torch.zeros_like(bd)
        P.apply(bd, z, nrhs)
        P.solve(bd, x, nrhs, rtol=1e-8)
        for k in range(nrhs):
            P.apply(bd[k].contiguous(), one)
            assert (z[k] - one).abs().max() <= 1e-12 * one.abs().max()
            r = b[k] - np.add.reduceat(M.val * x[k].cpu().numpy()[M.colind], M.rowptr[:-1])
            assert np.linalg.norm(r) <= 1.5e-8 * np.linalg.norm(b[k])
    finally:
        P.close()
