"""The network's training step and forward pass at the edges of their tiles: one
sample, around the 16 samples of a block, around the 128 samples of a gradient
split, and a buffer that is not 16-byte aligned, against the same in FP64.  Bars:
a chain of three 256-long FP32 sums, 256 u = 3e-5 of the largest magnitude."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _reference(wb, x, qt):
    w = torch.from_numpy(wb).double().requires_grad_(True)
    at, lay = 0, []
    for shape in ((32, 256), (256,), (256, 256), (256,), (256, 256), (256,)):
        lay.append(w[at:at + int(np.prod(shape))].view(shape))
        at += int(np.prod(shape))
    h = torch.relu(torch.from_numpy(x).double() @ lay[0] + lay[1])
    y = (torch.relu(h @ lay[2] + lay[3]) @ lay[4] + lay[5]).view(-1, 16, 16)
    q = 0.5 * (y + y.transpose(1, 2))
    loss = (q.reshape(len(x), -1) - torch.from_numpy(qt).double()).square().sum(1).mean()
    loss.backward()
    return q.detach().reshape(len(x), -1).numpy(), w.grad.numpy(), float(loss.detach())


@pytest.mark.parametrize("offset", (0, 1))
@pytest.mark.parametrize("n", (1, 15, 16, 17, 255, 256, 300, 1111))
def test_step_and_forward(n, offset):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    from paper_2109_05908_gb300 import learned
    rng = np.random.default_rng(n)
    wb = torch.from_numpy(learned.init_weights(1)).bfloat16().float().numpy()
    x = rng.standard_normal((n, 32)).astype(np.float32)
    qt = rng.standard_normal((n, 256)).astype(np.float32)

    def dev(a):
        t = torch.zeros(a.size + 1, dtype=torch.float32, device="cuda")[offset:offset + a.size]
        t.copy_(torch.from_numpy(a.ravel()))
        return t
    dw, dx, dq = dev(wb), dev(x), dev(qt)
    q, grad = torch.full((n, 256), 9.0, device="cuda"), torch.full((learned.NP,), 9.0, device="cuda")
    work, loss = torch.empty(A.mlp_sizes(n)[1] + 1, device="cuda")[offset:], torch.zeros(1, device="cuda")
    A.mlp_forward(dw.data_ptr(), dx.data_ptr(), n, q.data_ptr(), work.data_ptr())
    A.mlp_train_step(0, dw.data_ptr(), 0, 0, 0, 0.0, dx.data_ptr(), dq.data_ptr(), n, grad.data_ptr(), work.data_ptr(),
                     loss.data_ptr())
    rq, rg, rl = _reference(wb, x, qt)
    assert np.abs(q.cpu().numpy() - rq).max() <= 3e-5 * np.abs(rq).max()
    assert np.abs(grad.cpu().numpy() - rg).max() <= 3e-5 * np.abs(rg).max()
    assert abs(float(loss.item()) - rl) <= 3e-5 * rl
