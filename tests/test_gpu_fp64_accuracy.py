"""FP64 states of layered circuits against extended precision.

Tolerance: rotations applied entry by entry, as they were before their
diagonals were taken out into factors, leave these 240 states off by 8.2e-16
rms; products of rounded factors in FP64 by 8.3e-16."""
import numpy as np
import pytest

from paper_2609_23664_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_23664_gb300 import quwarp as Q  # noqa: E402


def _evolve(n, gates):
    psi = np.zeros(1 << n, dtype=np.clongdouble)
    psi[0] = 1
    idx = np.arange(1 << n)
    for g in gates:
        op, a, b = int(g["op"]), int(g["q0"]), int(g["q1"])
        if op == W.OP_CNOT:
            psi = psi[np.where((idx >> a) & 1, idx ^ (1 << b), idx)]
            continue
        half = np.longdouble(g["theta"]) / 2
        c, s = np.cos(half), np.sin(half)
        v = psi.reshape(1 << (n - 1 - a), 2, 1 << a)
        x, y = v[:, 0].copy(), v[:, 1].copy()
        if op == W.OP_RY:
            v[:, 0], v[:, 1] = c * x - s * y, s * x + c * y
        else:
            assert op == W.OP_RZ
            v[:, 0], v[:, 1] = (c - 1j * s) * x, (c + 1j * s) * y
        psi = v.reshape(-1)
    return psi


def test_rounding_of_layered_states():
    if np.finfo(np.longdouble).eps > 1e-18:
        pytest.skip("no extended precision on this host")
    n, err2 = 7, []
    eng = Q.Engine(0)
    for seed in range(60):
        tasks = W.vqe24_sweep(seed=seed, n=n, prefix_layers=6, n_tasks=4, max_suffix_layers=2, n_terms=20,
                              mode=W.MODE_SV_FP64)
        for t in tasks:
            t.want_state = True
        plan = Q.Plan(eng, Q.Workload(tasks)).run()
        for k, t in enumerate(tasks):
            d = plan.state(k, n, True).astype(np.clongdouble) - _evolve(n, t.gates)
            err2.append(float(np.sum(np.abs(d) ** 2)))
        plan.close()
    eng.close()
    rms = float(np.sqrt(np.mean(err2)))
    print("rms error of a state %.3g" % rms)
    assert rms <= 8.2e-16
