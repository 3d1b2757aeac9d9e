"""Long compensated tasks do share a launch: plans whose tasks all exceed the
pass limit run one wave per register size by default and one per task on an
engine that holds one chain at a time, in fewer launches, with the same bits."""
import numpy as np
import pytest

from paper_2609_23664_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_23664_gb300 import quwarp as Q  # noqa: E402


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("sizes,gates", [((14,), 1500), ((15, 17), 1000), ((16, 19), 800), ((21,), 600)])
def test_waves_and_bits(sizes, gates, shared):
    rng = np.random.default_rng(sum(sizes) + shared)
    count, tasks = 4, []
    for n in sizes:
        ham = W.random_pauli_hamiltonian(rng, n, 4)
        pre = W.random_circuit(rng, n, 150) if shared else None
        for i in range(count):
            tasks.append(W.Task(mode=W.MODE_SV_FP32, n=n, spans=([pre] if shared else []) + [W.random_circuit(rng, n, gates)],
                                terms=ham, want_state=i % 2 == 0))
    out, tuning = [], None
    for budget in (0, 1 << 16):  # default; less than one state
        eng = Q.Engine(0, task_budget_bytes=budget)
        if tuning:
            eng.load_tuning(tuning)
        plan = Q.Plan(eng, Q.Workload(tasks)).run()
        tuning = eng.tuning()
        rec = plan.cost_record()
        out.append((len(rec["wave_tiles"]), rec["kernel_launches"], [plan.energy(i) for i in range(len(tasks))],
                    [plan.state(i, t.n, False) for i, t in enumerate(tasks) if t.want_state]))
        plan.close()
        eng.close()
    assert (out[0][0], out[1][0]) == (len(sizes), count * len(sizes))
    assert out[0][1] + 6 * (count - 1) * len(sizes) <= out[1][1]  # a launch per pass, more than 6 each
    assert out[0][2] == out[1][2]
    assert all(np.array_equal(a, b) for a, b in zip(out[0][3], out[1][3]))
