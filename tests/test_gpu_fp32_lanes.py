"""Batched one-level applies of the mixed form at stage sizes on both sides of the
lines at which the lanes per row change (about 29,200, 14,600 and 7,300 rows): each
column against the same column alone, whose stages take the lanes of one vector.
(Not against an FP64 handle: a subdomain whose FP32 spectrum has a mu <= 0 by
rounding keeps that eigenvector at any tau, so the mixed form may have a coarse space.)

Bar: the parts are FP64 ones rounded to FP32 and a row sums at most K = 200 products
in FP32, so an entry is off by at most (K + 3) u32 sum |a| |x|; the inverse of an
M-matrix is positive and r is positive here, so the sums are the entries themselves,
and three such sums follow one another: 3 * 203 * 2^-24 = 3.7e-5 of the largest entry."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nrhs", [2, 8])
@pytest.mark.parametrize("m", [30, 60, 90, 130])
def test_fp32_lanes(m, nrhs):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    M = synth.laplace2d(m)
    M.val[M.val > 0] = 4.5
    part = (np.arange(m * m) // 100).astype(np.int32)
    r = torch.from_numpy(1.0 + np.abs(synth.rhs(M.n, 1, nrhs)).reshape(nrhs, M.n)).cuda()
    o = A.opts_default()
    o.precision = 1
    P = Preconditioner(DeviceMatrix(M), torch.from_numpy(part).cuda(), int(part[-1]) + 1, 1, 1e-17, o)
    try:
        z, one = torch.empty_like(r), torch.empty_like(r[0])
        P.apply(r, z, nrhs)
        for k in range(nrhs):
            P.apply(r[k].contiguous(), one)
            assert (z[k] - one).abs().max() <= 3.7e-5 * one.abs().max()
    finally:
        P.close()
