"""Stages of a single rotation without a phase (one RY or H), which run as a
general op: every position and register size from the smallest, FP32 compensated
and FP64, alone and between entangling gates, against the oracle; and the
arithmetic that the plan counts for such a stage.

Tolerance: one rounding of each amplitude (2^-24 of it) and 2^-38 of the
largest for the operations (FP64: 2^-50)."""
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


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n", [5, 6, 9, 13, 15])
@pytest.mark.parametrize("theta", [None, 0.7, np.pi / 2, 3.0, -2.0, 1e-9])
def test_one_rotation(eng, n, theta, fp64):
    rng = np.random.default_rng(n)
    for q in (0, n // 2, n - 1):
        one = (W.OP_H, q, 0, 0.0) if theta is None else (W.OP_RY, q, 0, theta)
        a, b = (int(v) for v in rng.choice(n, 2, replace=False))
        for gates in ([one], [(W.OP_CNOT, a, b, 0.0), one, (W.OP_CNOT, b, a, 0.0)]):
            gates = W.gates_from_list(gates)
            psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
            psi = psi.astype(np.complex128 if fp64 else np.complex64)
            st = torch.tensor(psi, device="cuda")
            Q.sv_apply_dev(eng, W.MODE_SV_FP64 if fp64 else W.MODE_SV_FP32, n, st.data_ptr(), gates)
            want = orc.sv_apply(n, psi.astype(np.complex128), gates)
            err = np.abs(st.cpu().numpy().astype(np.complex128) - want)
            big = np.abs(want).max()
            assert np.all(err <= (2.0 ** -50 * big if fp64 else 2.0 ** -24 * np.abs(want) + 2.0 ** -38 * big))


def test_counted_arithmetic(eng):
    # a two-term output (40 operations) and the split and rounding (10) on
    # each amplitude; with a phase, the stage's table (22 + 40 + 10)
    n = 10
    for phase, per_amplitude in ((False, 50), (True, 72)):
        g = [(W.OP_RY, 3, 0, 0.5)] + ([(W.OP_RZ, 3, 0, 0.2)] if phase else [])
        t = W.Task(mode=W.MODE_SV_FP32, n=n, spans=[W.gates_from_list(g)],
                   terms=W.random_pauli_hamiltonian(np.random.default_rng(0), n, 2))
        plan = Q.Plan(eng, Q.Workload([t])).run()
        assert plan.cost_record()["batch_alg_flops"] == per_amplitude * 2 ** n
        plan.close()
