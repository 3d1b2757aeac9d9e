"""Sampling around its block sizes: registers below, at and above one block of
4096 amplitudes, more blocks than threads of the offset scan, states on and
off a 16-byte boundary, long runs of zero amplitudes, uniforms at both ends.

A shot may differ from the FP64 CDF only where its uniform lies within 1e-6
of a step (FP32 probabilities are rounded to 2^-24 each); it always names an
outcome of nonzero probability."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("form", ["fp32", "fp32_off", "fp64"])
@pytest.mark.parametrize("n", [5, 11, 12, 13, 17, 21])
@pytest.mark.parametrize("shape", ["dense", "sparse", "ends"])
def test_shots_follow_the_cdf(eng, n, shape, form):
    rng = np.random.default_rng(10 * n + len(shape))
    dim = 1 << n
    psi = rng.normal(size=dim) + 1j * rng.normal(size=dim)
    if shape == "sparse":  # a few outcomes, most blocks empty
        keep = np.zeros(dim, bool)
        keep[rng.integers(0, dim, 6)] = True
        psi[~keep] = 0
    elif shape == "ends":
        psi[: dim // 3] = 0
        psi[dim - dim // 4:] = 0
    psi /= np.linalg.norm(psi)
    fp64 = form == "fp64"
    buf = torch.zeros(dim + 2, dtype=torch.complex128 if fp64 else torch.complex64, device="cuda")
    st = buf[1:1 + dim] if form == "fp32_off" else buf[:dim]
    st.copy_(torch.tensor(psi).to(st.dtype))
    assert (st.data_ptr() % 16 == 8) == (form == "fp32_off")
    u = np.concatenate([rng.random(300), [0.0, np.nextafter(1.0, 0.0), 0.5]])
    got = Q.sv_sample_dev(eng, W.MODE_SV_FP64 if fp64 else W.MODE_SV_FP32, n, st.data_ptr(), u).astype(np.int64)
    p = np.abs(st.cpu().numpy().astype(np.complex128)) ** 2
    cdf = np.cumsum(p) / p.sum()
    want = np.minimum(np.searchsorted(cdf, u, side="right"), np.nonzero(p)[0][-1])
    assert np.all(p[got] > 0)
    lo = np.where(got > 0, cdf[got - 1], 0.0)
    near = (u >= lo - 1e-6) & (u <= cdf[got] + 1e-6)
    assert np.all((got == want) | near)
    if shape == "sparse":
        steps = cdf[np.nonzero(p)[0]]
        clear = np.abs(u[:, None] - steps[None, :]).min(1) > 1e-6
        assert np.array_equal(got[clear], want[clear])
