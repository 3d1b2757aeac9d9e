"""Compensated rotations whose constants' error adds up: the same angle applied
thousands of times to every qubit (a Trotter circuit), and angles so small
that only the rotation's off-diagonal entry shows them.

Tolerance of the repeated angle: the chain rounds every amplitude once
(2^-24 of it), an operation errs by 2^-39 of its group's largest amplitude and
a stage runs at most nine of them on an amplitude (four rotations, a factor,
the split and the rounding), so 2^-24 |a| + 9 (stages) 2^-39 max|a|, with at
most three stages per repetition."""
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


@pytest.mark.parametrize("theta", [0.024139087302920074, 0.01048845545998558, 1.0689747013291277, 0.1, 2.9])
def test_repeated_angle(eng, theta):
    n, reps = 6, 5000
    # CNOTs are absorbed into the tile map, so every stage is one of rotations
    layer = [(W.OP_RY, q, 0, theta) for q in range(n)] + [(W.OP_CNOT, q, q + 1, 0.0) for q in range(n - 1)]
    gates = W.gates_from_list(layer * reps)
    psi = np.zeros(1 << n, dtype=np.complex64)
    psi[0] = 1
    st = torch.tensor(psi, device="cuda")
    Q.sv_apply_dev(eng, W.MODE_SV_FP32, n, st.data_ptr(), gates)
    want = orc.sv_apply(n, psi.astype(np.complex128), gates)
    err = np.abs(st.cpu().numpy().astype(np.complex128) - want)
    big = np.abs(want).max()
    print("max error / max|a| %.3g" % (err.max() / big))
    assert np.all(err <= 2.0 ** -24 * np.abs(want) + 9 * 3 * reps * 2.0 ** -39 * big)


@pytest.mark.parametrize("width", [1, 2, 4])
@pytest.mark.parametrize("theta", [1e-12, 1e-28, 1e-31, 1e-36])
def test_tiny_angles(eng, theta, width):
    n = 6
    gates = W.gates_from_list([(W.OP_RY, q, 0, theta) for q in range(width)])
    st = torch.zeros(1 << n, dtype=torch.complex64, device="cuda")
    st[0] = 1
    Q.sv_apply_dev(eng, W.MODE_SV_FP32, n, st.data_ptr(), gates)
    got = st.cpu().numpy()
    for q in range(width):
        # theta / 2, to a few FP32 roundings
        assert abs(float(got[1 << q].real) / (theta / 2) - 1) <= 2.0 ** -22
