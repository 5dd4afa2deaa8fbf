"""The network's loss: FP32 within a sample, FP64 over the samples.  With zero
weights the outputs are 0 and a sample's loss is the square of its one target entry:
4096^2 for one sample and 1 for the others is exact per sample, and a sum over samples
in FP32 drops the ones.  Bar: the rounding of the result to FP32, half a unit in the
last place."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 2, 16, 17, 40, 700])
@pytest.mark.parametrize("entry", [0, 17, 255])  # on the diagonal of the 16 x 16 output
def test_loss_over_samples(n, entry):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2109_05908_gb300 import amdd as A
    from paper_2109_05908_gb300 import learned
    w = torch.zeros(learned.NP, device="cuda")
    x = torch.ones((n, 32), device="cuda")
    q = torch.zeros((n, 256), device="cuda")
    q[:, entry] = 1.0
    q[n // 2, entry] = 4096.0
    grad, loss = torch.empty(learned.NP, device="cuda"), torch.zeros(1, device="cuda")
    work = torch.empty(A.mlp_sizes(n)[1], device="cuda")
    A.mlp_train_step(0, w.data_ptr(), 0, 0, 0, 0.0, x.data_ptr(), q.data_ptr(), n, grad.data_ptr(), work.data_ptr(),
                     loss.data_ptr())
    exact = (2.0 ** 24 + n - 1) / n
    assert abs(float(loss.item()) - exact) <= 0.5 * np.spacing(np.float32(exact))
