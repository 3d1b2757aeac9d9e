"""Cost-model gradient at batch sizes around its split over CTAs (one sample,
up to 100 CTAs of one, several per CTA, a ragged last CTA) against the FP64
oracle."""
import numpy as np
import pytest

from oracle import mlp_oracle as mo

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_23664_gb300 import quwarp as Q  # noqa: E402


@pytest.mark.parametrize("batch", [1, 2, 99, 100, 101, 256, 1023, 3001])
def test_gradient_batches(batch):
    rng = np.random.default_rng(batch)
    p = (0.2 * rng.normal(size=mo.N_PARAMS)).astype(np.float32)
    x = rng.normal(size=(batch, mo.N_IN)).astype(np.float32)
    t = rng.normal(size=batch).astype(np.float32)
    d = [torch.tensor(a, device="cuda") for a in (p, x, t)]
    loss = torch.zeros(1, device="cuda")
    grad = torch.zeros(mo.N_PARAMS, device="cuda")
    y = torch.zeros(batch, device="cuda")
    Q.mlp_loss_grad_dev(d[0].data_ptr(), d[1].data_ptr(), d[2].data_ptr(), batch, loss.data_ptr(), grad.data_ptr())
    Q.mlp_forward_dev(d[0].data_ptr(), d[1].data_ptr(), y.data_ptr(), batch)
    torch.cuda.synchronize()
    l_ref, g_ref = mo.loss_grad(p, x, t)
    y_ref, _ = mo.forward(p, x)
    # a hidden unit within FP32 rounding of a BF16 tie may round the other
    # way (2^-9 of one of 64 terms): bounded in the 2-norm over the batch
    assert np.linalg.norm(y.cpu().numpy() - y_ref) <= 1e-3 * np.linalg.norm(y_ref)
    assert abs(float(loss) - l_ref) <= 1e-3 * l_ref
    assert np.linalg.norm(grad.cpu().numpy() - g_ref) <= 2e-3 * np.linalg.norm(g_ref)
