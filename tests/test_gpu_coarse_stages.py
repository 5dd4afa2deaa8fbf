"""The coarse solve by substructuring at the edges of its plan: one part, two
and three stages, several components, dense blocks of a partial selection, one
to eight vectors.  M^{-1} r against the oracle's apply to the suite's bar of
1e-10 (FP64 rounding of two exact solves of well-conditioned problems)."""
import numpy as np
import pytest

import synth
from oracle import amdd_oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _lap(m, box, tau):
    part = synth.box_partition_2d(m, box)
    return synth.laplace2d(m), part, int(part.max()) + 1, tau


def _blocks(m, nb):
    M, part = synth.disjoint_blocks(m, nb)
    return M, np.asarray(part, np.int32), int(np.max(part)) + 1, 50.0


CASES = {
    "one_part_81": lambda: _lap(9, 3, 50.0),
    "two_stages_100": lambda: _lap(10, 5, 50.0),
    "two_stages_1089": lambda: _lap(33, 11, 50.0),
    "three_stages_1225": lambda: _lap(35, 7, 50.0),
    "dense_blocks_partial": lambda: _lap(32, 8, 0.5),
    "components": lambda: _blocks(12, 3),
}


@pytest.mark.parametrize("name", CASES)
def test_apply_matches_oracle(name):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    M, part, N, tau = CASES[name]()
    S = O.setup(M, part, N, 1, tau)
    P = Preconditioner(DeviceMatrix(M), torch.from_numpy(np.ascontiguousarray(part, np.int32)).cuda(), N, 1, tau)
    try:
        assert P.info().n_C == S.nC
        for nrhs in (1, 3, 8, 11):
            r = synth.rhs(M.n, 5, nrhs).reshape(nrhs, M.n)
            rd = torch.from_numpy(r).cuda()
            zd = torch.empty_like(rd)
            P.apply(rd, zd, nrhs)
            z = zd.cpu().numpy()
            for k in range(nrhs):
                zo = O.apply(S, r[k])
                assert np.linalg.norm(z[k] - zo) <= 1e-10 * np.linalg.norm(zo), (nrhs, k)
    finally:
        P.close()
