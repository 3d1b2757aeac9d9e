"""Rounding of the cost model's gradient: the median over batches of 256 of
its distance from the FP64 oracle, in the 2-norm.  Tolerance: CTAs of 32
samples, their partials added one by one, left 7.0e-8 (the median leaves out
the batches in which a hidden unit rounds to the other BF16 neighbour)."""
import numpy as np
import pytest

from oracle import mlp_oracle as mo

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_23664_gb300 import quwarp as Q  # noqa: E402


def test_gradient_rounding():
    batch, errs = 256, []
    for seed in range(15):
        rng = np.random.default_rng(seed)
        p = (0.2 * rng.normal(size=mo.N_PARAMS)).astype(np.float32)
        x = rng.normal(size=(batch, mo.N_IN)).astype(np.float32)
        t = rng.normal(size=batch).astype(np.float32)
        d = [torch.tensor(a, device="cuda") for a in (p, x, t)]
        loss = torch.zeros(1, device="cuda")
        grad = torch.zeros(mo.N_PARAMS, device="cuda")
        Q.mlp_loss_grad_dev(d[0].data_ptr(), d[1].data_ptr(), d[2].data_ptr(), batch, loss.data_ptr(), grad.data_ptr())
        torch.cuda.synchronize()
        ref = mo.loss_grad(p, x, t)[1]
        errs.append(np.linalg.norm(grad.cpu().numpy() - ref) / np.linalg.norm(ref))
    print("median %.3g" % np.median(errs))
    assert np.median(errs) <= 7.0e-8
