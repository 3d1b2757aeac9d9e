"""FP64 rotation stages (unnormalized rotations, one factor per amplitude):
angles around 0, 45, 90 and 180 degrees, one to six qubits of a stage, with and
without phases, registers of one tile and of several.

Tolerance: at most 8 roundings of 2^-53 per amplitude and operation over fewer
than 16 operations: 2^-46 of the largest amplitude."""
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


@pytest.mark.parametrize("n", [5, 11, 14])
@pytest.mark.parametrize("width", [1, 2, 4, 5, 6])
@pytest.mark.parametrize("theta", [0.0, 1e-14, np.pi / 2, np.pi / 2 - 1e-12, np.pi, np.pi + 1e-9, 2 * np.pi, 4.4])
def test_rotation_stages(eng, theta, width, n):
    rng = np.random.default_rng(17 * n + width)
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    g = []
    for q in range(min(width, n)):
        g.append((W.OP_RY, n - 1 - q, 0, theta))
        if q % 2:
            g.append((W.OP_RZ, n - 1 - q, 0, float(rng.uniform(0, 6.28))))
    g += [(W.OP_CNOT, 0, n - 1), (W.OP_RY, 0, 0, -theta)]
    gates = W.gates_from_list(g)
    st = torch.tensor(psi, device="cuda")
    Q.sv_apply_dev(eng, W.MODE_SV_FP64, n, st.data_ptr(), gates)
    want = orc.sv_apply(n, psi.copy(), gates)
    assert np.abs(st.cpu().numpy() - want).max() <= 2.0 ** -46 * np.abs(want).max()
