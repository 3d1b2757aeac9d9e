"""Compensated stages at the edges of their group grid: states scaled far up
and down (the grid and its low parts would leave the FP32 range), rotations at
and around 45 and 90 degrees (exchanged halves, exact quotients), zero groups,
every partial rotation stage, and non-finite amplitudes.

Tolerance: the chain rounds every amplitude once (2^-24 relative of it) and a
register operation errs by 2^-39 of its group's largest amplitude, so with up
to 64 operations an amplitude is off by at most 2^-24 |a| + 2^-33 max|a|."""
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


def _run(eng, n, psi, gates):
    st = torch.tensor(psi, device="cuda")
    Q.sv_apply_dev(eng, W.MODE_SV_FP32, n, st.data_ptr(), gates)
    return st.cpu().numpy()


def _gates(n, angles, phases):
    g = []
    for q in range(n):
        if angles[q] is not None:
            g.append((W.OP_RY, q, 0, angles[q]))
        if phases[q] is not None:
            g.append((W.OP_RZ, q, 0, phases[q]))
    return W.gates_from_list(g)


@pytest.mark.parametrize("scale", [0, -70, -95, -110, 100, 118])
@pytest.mark.parametrize("mix", ["rotations", "general"])
def test_scaled_states(eng, scale, mix):
    n = 9
    rng = np.random.default_rng(700 + scale)
    psi = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)).astype(np.complex64)
    psi[:48] = 0  # whole groups and parts of groups of zeros
    if mix == "rotations":
        gates = _gates(n, rng.uniform(0, 6.28, n), rng.uniform(0, 6.28, n))
    else:
        gates = W.random_circuit(rng, n, 40)
    got = _run(eng, n, (psi * np.float32(2.0) ** scale).astype(np.complex64), gates)
    want = orc.sv_apply(n, psi.astype(np.complex128), gates)
    got = got.astype(np.complex128) * 2.0 ** -scale
    # numbers stored below 2^-126 round to multiples of 2^-149, remainders
    # at every one of at most 64 stages
    floor = 64 * 2.0 ** (-149 - scale) if scale < 0 else 0.0
    err = np.abs(got - want)
    assert np.all(err <= 2.0 ** -24 * np.abs(want) + 2.0 ** -33 * np.abs(want).max() + floor)


@pytest.mark.parametrize("theta", [0.0, 1e-12, 1e-5, np.pi / 2, np.pi / 2 + 2.0 ** -30, np.pi / 2 - 2.0 ** -25, np.pi,
                                   np.pi - 1e-9, 2 * np.pi, 3.0, -1.25])
@pytest.mark.parametrize("width", [1, 2, 3, 4, 7])
def test_rotation_angles_and_partial_stages(eng, theta, width):
    n = 8
    rng = np.random.default_rng(31 + width)
    psi = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)).astype(np.complex64)
    angles = [theta if q < width else None for q in range(n)]
    phases = [float(rng.uniform(0, 6.28)) if q < width and q % 2 == 0 else None for q in range(n)]
    gates = _gates(n, angles, phases)
    got = _run(eng, n, psi, gates).astype(np.complex128)
    want = orc.sv_apply(n, psi.astype(np.complex128), gates)
    err = np.abs(got - want)
    assert np.all(err <= 2.0 ** -24 * np.abs(want) + 2.0 ** -33 * np.abs(want).max())


def test_non_finite_amplitudes_stay_in_their_groups(eng):
    n = 10
    rng = np.random.default_rng(5)
    psi = (rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)).astype(np.complex64)
    gates = W.gates_from_list([(W.OP_RY, q, 0, 0.3 + q) for q in range(2)])
    want = orc.sv_apply(n, psi.astype(np.complex128), gates)
    for bad in (np.nan, np.inf):
        p = psi.copy()
        p[517] = bad
        got = _run(eng, n, p, gates)
        hit = np.arange(1 << n) // 4 == 517 // 4  # the four amplitudes that mix with it
        assert not np.isfinite(got[hit]).any()
        assert np.all(np.abs(got[~hit] - want[~hit]) <= 1e-6 * np.abs(want).max())
