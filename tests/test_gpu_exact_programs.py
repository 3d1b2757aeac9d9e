"""Gate lists that only permute amplitudes and multiply them by +-1 and +-i:
applied to the caller's state and in a plan they give the permuted state to
the bit, from one tile to many, FP32 and FP64, tiny and huge amplitudes among
ordinary ones; a plan's permutations of a register that fits one
tile run in one."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2609_23664_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_23664_gb300 import quwarp as Q  # noqa: E402

ONE = [W.OP_X, W.OP_Y, W.OP_Z, W.OP_S, W.OP_SDG]
TWO = [W.OP_CNOT, W.OP_CZ, W.OP_SWAP]


@pytest.fixture(scope="module")
def eng():
    e = Q.Engine(0)
    yield e
    e.close()


def _gates(rng, n, count, ops):
    g = []
    for _ in range(count):
        op = int(rng.choice(ops))
        a, b = (int(v) for v in rng.choice(n, 2, replace=False))
        g.append((op, a, b if op in TWO else 0, 0.0))
    return W.gates_from_list(g)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n", [5, 9, 12, 13, 14, 17])
@pytest.mark.parametrize("kind", ["permutations", "all"])
def test_states_to_the_bit(eng, n, fp64, kind):
    rng = np.random.default_rng(n)
    gates = _gates(rng, n, 80, [W.OP_X, W.OP_CNOT, W.OP_SWAP] if kind == "permutations" else ONE + TWO)
    psi = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)) * 10.0 ** rng.uniform(-12, 8, 1 << n)
    psi = psi.astype(np.complex128 if fp64 else np.complex64)
    st = torch.tensor(psi, device="cuda")
    Q.sv_apply_dev(eng, W.MODE_SV_FP64 if fp64 else W.MODE_SV_FP32, n, st.data_ptr(), gates)
    want = orc.sv_apply(n, psi.astype(np.complex128), gates)
    assert np.array_equal(st.cpu().numpy().astype(np.complex128), want)


@pytest.mark.parametrize("fp64", [False, True])
def test_plans_take_one_tile(eng, fp64):
    n = 13
    rng = np.random.default_rng(1)
    gates = _gates(rng, n, 400, [W.OP_X, W.OP_CNOT, W.OP_SWAP])
    mode = W.MODE_SV_FP64 if fp64 else W.MODE_SV_FP32
    t = W.Task(mode=mode, n=n, spans=[gates], terms=W.random_pauli_hamiltonian(rng, n, 3), want_state=True)
    plan = Q.Plan(eng, Q.Workload([t])).run()
    assert plan.cost_record()["wave_tiles"][0][0] == 13
    psi = np.zeros(1 << n, dtype=np.complex128)
    psi[0] = 1
    want = orc.sv_apply(n, psi, gates)
    assert np.array_equal(plan.state(0, n, fp64).astype(np.complex128), want)
    plan.close()
