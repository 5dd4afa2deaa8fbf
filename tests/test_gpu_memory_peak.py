"""Setups within the device memory that they took when the local solves were the dense
triangles of A_ii: the peak of that form, measured on these problems, as mem_budget.
And a batched solve on a handle that has served single vectors before, whose
batched work vectors are allocated then."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# bytes: 3D elasticity, 9^3 elements in boxes of 5 (tau, precision), 256 x 256 Laplacian in 256 boxes (mixed, one level)
PEAK = {
    ("elas", 1e-17, 0): 391077980, ("elas", 1e-17, 1): 169675404, ("elas", 1e-17, 2): 356092456,
    ("elas", 0.5, 0): 443541816, ("elas", 0.5, 1): 187711312, ("elas", 0.5, 2): 397418344,
    ("lap", 1e-17, 1): 1339671052,
}


def _problem(what):
    if what == "lap":
        return synth.laplace2d(256), synth.box_partition_2d(256, 16)
    M, _, xyz = synth.elasticity3d(9, layer=2)
    return M, synth.box_partition_dofs(xyz, (5, 5, 5))


@pytest.mark.parametrize("what,tau,precision", list(PEAK))
def test_setup_within_the_former_peak(what, tau, precision):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    M, part = _problem(what)
    o = A.opts_default()
    o.precision = precision
    o.mem_budget = PEAK[what, tau, precision]
    P = Preconditioner(DeviceMatrix(M), torch.from_numpy(np.asarray(part, np.int32)).cuda(), int(part.max()) + 1, 1, tau, o)
    try:
        assert P.info().device_bytes_peak <= PEAK[what, tau, precision]
    finally:
        P.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_single_vectors_between_batched_ones(precision):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    M = synth.laplace2d(48)
    part = synth.box_partition_2d(48, 12)
    o = A.opts_default()
    o.precision = precision
    P = Preconditioner(DeviceMatrix(M), torch.from_numpy(np.asarray(part, np.int32)).cuda(), 16, 1, 50.0, o)
    try:
        b = torch.from_numpy(synth.rhs(M.n, 1, 8).reshape(8, M.n)).cuda()
        first, again, z = torch.empty_like(b[0]), torch.empty_like(b[0]), torch.empty_like(b)
        P.apply(b[0].contiguous(), first)
        P.apply(b, z, 8)
        P.apply(b[0].contiguous(), again)
        assert torch.equal(first, again)
        assert (z[0] - first).abs().max() <= (1e-12 if precision == 0 else 1e-4) * first.abs().max()
    finally:
        P.close()
