"""Applies and solves with a coarse space on the caller's own stream: the coarse solve runs
beside the local solves on a second stream of the handle, between what the caller
enqueued before and after.  Repeated calls whose input is written on that stream just
before, and whose result is read on it just after, without any other synchronisation,
give the bits of a call on settled data; so do two handles on two streams."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tau,precision", [(50.0, 0), (50.0, 1), (0.5, 0)])
def test_repeated_calls_on_own_streams(tau, precision):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    from paper_2109_05908_gb300.device import DeviceMatrix, Preconditioner
    M = synth.laplace2d(40)
    part = torch.from_numpy(synth.box_partition_2d(40, 10)).cuda()
    dM = DeviceMatrix(M)
    r = torch.from_numpy(synth.rhs(M.n, 1, 6).reshape(6, M.n)).cuda()
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    P = []
    for s in streams:
        with torch.cuda.stream(s):
            o = A.opts_default()
            o.precision = precision
            P.append(Preconditioner(dM, part, 16, 1, tau, o, stream=s.cuda_stream))
    try:
        assert P[0].info().n_C > 0
        want = torch.empty_like(r)
        for k in range(6):
            P[0].apply(r[k], want[k])
        torch.cuda.synchronize()
        big = torch.randn(8_000_000, device="cuda")
        for turn in range(12):
            for s, p in zip(streams, P):
                with torch.cuda.stream(s):
                    k = turn % 6
                    junk = big * 2.0  # work ahead of the input on the stream
                    x = r[k] * 2.0 * 0.5 + 0.0 * junk[: M.n].double()
                    z = torch.full_like(x, 7.0)
                    p.apply(x, z)
                    got = z * 1.0
                    z.fill_(3.0)
                    sol = torch.zeros_like(x)
                    st = p.solve(x, sol, rtol=1e-8)
                assert torch.equal(got, want[k]) and st.converged == 1
    finally:
        for p in P:
            p.close()
