"""The remainder arrays of boundaries that share a launch count against the
task budget: with a budget that would just hold every task's state, the
arrays push a task into a second wave."""
import numpy as np
import pytest

from energy_tol import FP32_ENERGY_TOL, energy_error
from oracle import oracle as orc
from paper_2609_23664_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_23664_gb300 import quwarp as Q  # noqa: E402


def test_boundary_remainders_count():
    rng = np.random.default_rng(3)
    tasks = []
    for _ in range(4):  # four boundaries of 16 qubits and several passes, two tasks each
        pre = W.random_circuit(rng, 16, 150)
        for _ in range(2):
            tasks.append(W.Task(mode=W.MODE_SV_FP32, n=16, spans=[pre, W.random_circuit(rng, 16, 12)],
                                terms=W.random_pauli_hamiltonian(rng, 16, 3)))
    for _ in range(8):
        tasks.append(W.Task(mode=W.MODE_SV_FP32, n=18, spans=[W.random_circuit(rng, 18, 12)],
                            terms=W.random_pauli_hamiltonian(rng, 18, 3)))
    states = 8 * (8 << 16) + 8 * (8 << 18)  # every task's state; the remainders take 4 x 512 KB more
    waves = []
    for budget in (states, states + 4 * (8 << 16)):
        eng = Q.Engine(0, task_budget_bytes=budget)
        plan = Q.Plan(eng, Q.Workload(tasks), delta_frac=0.0).run()
        ex = plan.explain()["decisions"]
        assert [d["decision"] for d in ex] == ["REUSE"] * 4
        waves.append(len(plan.cost_record()["wave_tiles"]))
        for i in range(0, len(tasks), 3):
            ref = orc.run_task(tasks[i])
            assert energy_error(plan.energy(i)[0], ref["energy"], tasks[i].terms, tasks[i].n) <= FP32_ENERGY_TOL, i
        plan.close()
        eng.close()
    assert waves == [3, 2]
