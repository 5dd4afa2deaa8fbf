"""Partial selections whose kept eigenvector is spread evenly over a large
subdomain: n unknowns of one subdomain, not coupled to each other, around one
unknown of another.  With A = [[I, -a], [-a^T, n/(1 - mu)]], a all ones, the
eigenproblem of the first subdomain has the matrix I - (1 - mu) v v^T, v = 1/sqrt(n):
one eigenvalue mu, all others 1, and every pair of rows has a cosine of about
(1 - mu^2)/n only, so an eigenvector solver that leaves small couplings of long
rows alone must not leave these.

Bars on the sine of the angle between the coarse block and the oracle's: the
suite's 1e-8 in FP64; 1e-3 with FP32 local work on the FP64 splitting (T rounded
to n u32 |T| = 7e-5, gap 0.55); with the FP32 splitting twice the suite's
4 u32 kappa_X for such an apply (gap 0.55)."""
import numpy as np
import pytest

import synth
from oracle import amdd_oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def star(n, mu):
    i, hub = np.arange(n), np.full(n, n)
    M = synth._csr_from_coo(n + 1, np.concatenate([i, i, hub, [n]]), np.concatenate([i, hub, i, [n]]),
                            np.concatenate([np.ones(n), -np.ones(2 * n), [n / (1.0 - mu)]]))
    return M, (np.arange(n + 1) == n).astype(np.int32)


@pytest.mark.parametrize("precision", [0, 1, 2])
@pytest.mark.parametrize("n,mu", [(1100, 0.01), (900, 0.45), (400, 0.45)])
def test_spread_eigenvector(n, mu, precision):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    M, part = star(n, mu)
    S = O.setup(M, part, 2, 1, 0.5, eps=2.0 ** -23 if precision == 1 else 2.0 ** -52)
    s = S.subs[0]
    assert s.p == 1
    kappa = s.sigma.max() / s.sigma.min()
    bar = {0: 1e-8, 1: 2 * 4 * 2.0 ** -24 * kappa, 2: 1e-3}[precision]
    o = A.opts_default()
    o.precision = precision
    P = Preconditioner(DeviceMatrix(M), torch.from_numpy(part).cuda(), 2, 1, 0.5, o)
    try:
        assert P.info().n_C == S.nC
        z = A.get_coarse_block(P.h, 0)
        assert z.shape == (1, n)
        z = z[0] / np.linalg.norm(z)
        u = s.Z[:n, 0] / np.linalg.norm(s.Z[:n, 0])
        assert np.linalg.norm(z - u * (u @ z)) <= bar
    finally:
        P.close()
