"""Energies and norms of unnormalized FP32 states: amplitudes whose squares
fit FP32 while the sums over a warp do not, and ones near its lower end.  The
states are powers of two times small whole numbers, so every product and sum
is exact."""
import numpy as np
import pytest

from paper_2609_23664_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_23664_gb300 import quwarp as Q  # noqa: E402


@pytest.mark.parametrize("n", [5, 9, 14, 18])
@pytest.mark.parametrize("scale", [-50, 0, 57, 59])
def test_scaled_states(n, scale):
    rng = np.random.default_rng(n)
    v = (rng.integers(1, 3, 1 << n) + 1j * rng.integers(-1, 2, 1 << n)).astype(np.complex64)
    st = torch.tensor((v * np.float32(2.0) ** scale).astype(np.complex64), device="cuda")
    terms = W.random_pauli_hamiltonian(rng, n, 6)
    terms["coef"] = 2.0 ** rng.integers(-3, 1, 6)
    terms["xmask"][0] = 0
    eng = Q.Engine(0)
    e, norm = Q.sv_energy_dev(eng, W.MODE_SV_FP32, n, st.data_ptr(), terms)
    eng.close()
    x, i = v.astype(np.complex128), np.arange(1 << n)
    want = 0.0
    for t in terms:
        m, z = int(t["xmask"]), int(t["zmask"])
        sign = 1 - 2 * (np.array([bin(k & z).count("1") for k in range(1 << n)]) & 1)
        want += float(t["coef"]) * float(np.real(1j ** (bin(m & z).count("1") % 4) * np.sum(np.conj(x[i ^ m]) * sign * x)))
    n2 = float(np.sum(np.abs(x) ** 2))
    assert norm == n2 * 4.0 ** scale
    assert abs(e - want / n2) <= 2.0 ** -50 * max(1.0, abs(want / n2))
