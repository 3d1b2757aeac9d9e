"""qw_costmodel_train with a shorter last batch, whose gradient may take more
CTAs than a full one's, against the same steps in FP64.

Tolerance: gradients agree to 2e-3 of their norm (BF16 ties, as for single
batches), and Adam's first steps move every parameter by about lr whatever its
gradient's size, so parameters with a gradient below 2e-3 of the typical one
(0.2 % of them) may step the other way: 2 lr sqrt(0.002) = 0.09 of the
distance travelled.  A last batch with a damaged gradient is off by about its
share of the steps, a half."""
import subprocess

import numpy as np
import pytest

from oracle import mlp_oracle as mo

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_23664_gb300 import quwarp as Q  # noqa: E402

# the order in which training visits its rows: the generator that draws the
# initial weights shuffles them, anew each epoch
ORDER = r"""
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>
int main(int, char **v) {
  std::mt19937_64 rng(strtoull(v[1], 0, 10));
  const int n = atoi(v[2]), epochs = atoi(v[3]);
  std::uniform_real_distribution<double> U(-1, 1);
  for (int i = 0; i < 12 * 64 + 64 * 64 + 64; i++) U(rng);
  std::vector<uint32_t> perm(n);
  for (int i = 0; i < n; i++) perm[i] = i;
  for (int e = 0; e < epochs; e++) {
    std::shuffle(perm.begin(), perm.end(), rng);
    for (uint32_t p : perm) printf("%u\n", p);
  }
}
"""


@pytest.fixture(scope="module")
def order(tmp_path_factory):
    d = tmp_path_factory.mktemp("order")
    (d / "order.cpp").write_text(ORDER)
    subprocess.run(["g++", "-O1", "-std=c++17", "-o", str(d / "order"), str(d / "order.cpp")], check=True)
    return lambda seed, n, epochs: np.array(
        subprocess.run([str(d / "order"), str(seed), str(n), str(epochs)], check=True, capture_output=True,
                       text=True).stdout.split(), dtype=np.int64).reshape(epochs, n)


@pytest.mark.parametrize("batch,last", [(256, 87), (256, 100), (256, 173), (256, 200), (101, 100), (256, 256), (64, 1)])
def test_training_with_a_shorter_last_batch(order, batch, last):
    n, epochs, lr, seed = batch + last, 2, 1e-3, 40 + last
    rng = np.random.default_rng(seed)
    x = rng.normal(size=(n, mo.N_IN)).astype(np.float32)
    t = (12 + np.tanh(x[:, 0]) + 0.5 * x[:, 1]).astype(np.float32)
    eng = Q.Engine(0)
    eng.costmodel_train(x, t, epochs=0, batch=batch, lr=lr, seed=seed)
    p0, mean, scale = eng.costmodel_get()
    loss = eng.costmodel_train(x, t, epochs=epochs, batch=batch, lr=lr, seed=seed)
    got = eng.costmodel_get()[0].astype(np.float64)
    eng.close()
    xn = (x - mean) / scale
    p, m, v, step = p0.astype(np.float64), 0.0, 0.0, 0
    for perm in order(seed, n, epochs):
        for b0 in range(0, n, batch):
            rows = perm[b0:b0 + batch]
            step += 1
            g = mo.loss_grad(p.astype(np.float32), xn[rows], t[rows])[1]
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            p = p - lr * (m / (1 - 0.9 ** step)) / (np.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    assert step == 2 * epochs
    assert np.linalg.norm(got - p) <= 0.1 * np.linalg.norm(p - p0)
    l_ref = mo.loss_grad(got.astype(np.float32), xn, t)[0]
    assert abs(loss - l_ref) <= 1e-3 * l_ref
