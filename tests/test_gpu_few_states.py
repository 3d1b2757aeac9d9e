"""Plans with few compensated states take tiles of 2^12 amplitudes where the
tuner, which times many states, prefers wider ones; where one of them keeps
its remainder all do.  Results against the oracle on both sides of the rule."""
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


@pytest.fixture(scope="module")
def eng():
    e = Q.Engine(0)
    # 16 qubits: a shape the tuner might choose for many states
    Q.Plan(e, Q.Workload(_tasks(16, 1, 30))).close()
    rec = e.tuning()
    shape = dict([t for t in rec["tiles"] if t["n"] == 16 and t["arith"] == 1][0], k=13, b=4)
    rec["tiles"] = [dict(shape, mix=m) for m in (0, 1)]  # for either gate mix
    e.close()
    e = Q.Engine(0)
    e.load_tuning(rec)
    yield e
    e.close()


def _tasks(n, count, gates):
    rng = np.random.default_rng(n + count)
    ham = W.random_pauli_hamiltonian(rng, n, 4)
    return [W.Task(mode=W.MODE_SV_FP32, n=n, spans=[W.random_circuit(rng, n, g)], terms=ham)
            for g in (gates if isinstance(gates, list) else [gates] * count)]


def _check(plan, tasks, step):
    for i in range(0, len(tasks), step):
        ref = orc.run_task(tasks[i])
        assert energy_error(plan.energy(i)[0], ref["energy"], tasks[i].terms, tasks[i].n) <= FP32_ENERGY_TOL, i


@pytest.mark.parametrize("count,tile", [(1, 12), (64, 12), (65, 13)])
def test_tiles_follow_the_number_of_states(eng, count, tile):
    tasks = _tasks(16, count, 30)
    plan = Q.Plan(eng, Q.Workload(tasks), reuse=0).run()
    assert plan.cost_record()["wave_tiles"][0][0] == tile
    _check(plan, tasks, 16)
    plan.close()


def test_one_wave_for_chains_and_others(eng):
    tasks = _tasks(16, 4, [40, 500, 60, 450])
    plan = Q.Plan(eng, Q.Workload(tasks), reuse=0).run()
    assert len(plan.cost_record()["wave_tiles"]) == 1
    _check(plan, tasks, 1)
    plan.close()
