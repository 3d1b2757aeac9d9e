"""Compensated passes around the tile count where every stage group gets a
thread of its own (at most 128 tiles), against the oracle.

Tolerance: one rounding of each amplitude, and 2^-39 of the largest for each of
at most 64 operations on it, as for other compensated chains."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2609_23664_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_23664_gb300 import quwarp as Q  # noqa: E402


@pytest.fixture(scope="module")
def eng():
    e = Q.Engine(0)
    yield e
    e.close()


@pytest.mark.parametrize("n", [5, 8, 11, 12, 13, 18, 19, 20])
def test_call(eng, n):
    rng = np.random.default_rng(n)
    gates = W.random_circuit(rng, n, 60)
    psi = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)).astype(np.complex64)
    st = torch.tensor(psi, device="cuda")
    Q.sv_apply_dev(eng, W.MODE_SV_FP32, n, st.data_ptr(), gates)
    want = orc.sv_apply(n, psi.astype(np.complex128), gates)
    err = np.abs(st.cpu().numpy().astype(np.complex128) - want)
    assert np.all(err <= 2.0 ** -24 * np.abs(want) + 2.0 ** -33 * np.abs(want).max())
