"""Long compensated tasks that share a persistent launch, against the same
tasks one after another: an engine whose task budget holds one chain at a
time runs them pass by pass.  Both run the same passes on the same remainders,
so states and energies agree bit for bit; a few are checked against the
oracle.  Registers from one pass per tile to several sizes in one plan, tasks
that keep their state and tasks from the pool, with and without boundaries
(whose passes share a launch while their remainders fit)."""
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


def _tasks(rng, sizes, shared):
    tasks = []
    for n in sizes:
        ham = W.random_pauli_hamiltonian(rng, n, 6)
        pre = W.random_circuit(rng, n, 120) if shared else None
        for i in range(5):
            spans = ([pre] if shared else []) + [W.random_circuit(rng, n, int(rng.integers(260, 420)))]
            tasks.append(W.Task(mode=W.MODE_SV_FP32, n=n, spans=spans, terms=ham, want_state=i % 3 == 0))
    return tasks


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("sizes", [(14,), (15, 17), (16, 18, 21)])
def test_shared_launch_equals_one_by_one(sizes, shared):
    rng = np.random.default_rng(sum(sizes) + shared)
    tasks = _tasks(rng, sizes, shared)
    out = []
    for budget in (0, 1 << 16):  # default; less than one state
        eng = Q.Engine(0, task_budget_bytes=budget)
        if out:
            eng.load_tuning(tuning)
        plan = Q.Plan(eng, Q.Workload(tasks)).run()
        tuning = eng.tuning()
        out.append(([plan.energy(i) for i in range(len(tasks))],
                    [plan.state(i, t.n, False) if t.want_state else None for i, t in enumerate(tasks)]))
        plan.close()
        eng.close()
    for i, t in enumerate(tasks):
        assert out[0][0][i] == out[1][0][i], i
        if t.want_state:
            assert np.array_equal(out[0][1][i], out[1][1][i]), i
    for i in range(0, len(tasks), 4):
        ref = orc.run_task(tasks[i])
        assert energy_error(out[0][0][i][0], ref["energy"], tasks[i].terms, tasks[i].n) <= FP32_ENERGY_TOL, i
