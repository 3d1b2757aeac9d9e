"""Grouped energy terms: Hamiltonians whose flip masks span fewer or exactly
four dimensions, share spans, flip bit 0 alone or with others (the pair of a
16-byte load), repeat one mask with many phases, on the smallest registers
and around the block sizes, on states on and off a 16-byte boundary, and for
registers whose blocks take several runs of representatives.

Tolerance: FP32 products (2^-24 relative each) summed over at most 32 pairs in
FP32 and then in pairs of FP32: 4e-7 of the energy's typical size, the bound
of the kernel-level energy tests; FP64 1e-12."""
import numpy as np
import pytest

from energy_tol import energy_error
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


def _terms(rng, n, kind):
    full = (1 << n) - 1
    if kind == "span":  # every combination of five masks, two phases each
        base = [int(m) for m in rng.integers(1, full + 1, 5)]
        masks = []
        for c in range(32):
            m = 0
            for i in range(5):
                m ^= base[i] if c >> i & 1 else 0
            masks += [m, m]
    elif kind == "bit0":
        masks = [1, 1, 0, 2 & full, 3 & full, 1] + [int(m) | 1 for m in rng.integers(0, full + 1, 6)]
        masks += [m ^ 1 for m in masks]
    elif kind == "few":
        masks = [full]
    elif kind == "high":  # neighbours in the highest bits, every class
        masks = [int(m) << max(0, n - 4) for m in range(16)] + [1 << (n - 1) | 1]
    else:
        masks = [int(m) for m in rng.integers(0, full + 1, 23)]
    t = np.zeros(len(masks), dtype=W.TERM_DTYPE)
    t["xmask"] = [m & full for m in masks]
    t["zmask"] = rng.integers(0, full + 1, len(masks))
    t["coef"] = rng.normal(size=len(masks))
    return t


@pytest.mark.parametrize("kind", ["span", "bit0", "few", "high", "random"])
@pytest.mark.parametrize("n", [5, 6, 9, 13, 14, 19, 24])
@pytest.mark.parametrize("form", ["fp32", "fp32_off", "fp64"])
def test_groups_match_the_oracle(eng, form, n, kind):
    if n == 24 and (kind not in ("high", "random") or form == "fp64"):
        pytest.skip("one class structure per form is enough at this size")
    rng = np.random.default_rng(100 * n + len(kind))
    psi = rng.normal(size=1 << n) + 1j * rng.normal(size=1 << n)
    psi *= 0.8 / np.linalg.norm(psi)
    fp64 = form == "fp64"
    if not fp64:
        psi = psi.astype(np.complex64).astype(np.complex128)
    pad = 1 if form == "fp32_off" else 2  # FP32: one element off the allocation's 16-byte boundary, or on it
    buf = torch.zeros((1 << n) + 2, dtype=torch.complex128 if fp64 else torch.complex64, device="cuda")
    st = buf[pad:pad + (1 << n)]
    st.copy_(torch.tensor(psi).to(st.dtype))
    assert (st.data_ptr() % 16 == 8) == (form == "fp32_off")
    terms = _terms(rng, n, kind)
    mode = W.MODE_SV_FP64 if fp64 else W.MODE_SV_FP32
    e, nr = Q.sv_energy_dev(eng, mode, n, st.data_ptr(), terms)
    out = torch.zeros(2, dtype=torch.float64, device="cuda")
    Q.sv_energy_noalloc_dev(mode, n, st.data_ptr(), terms, out.data_ptr())
    e_ref, n_ref, _ = orc.energy(n, psi, terms)
    for got, norm in ((e, nr), out.tolist()):
        if fp64:
            assert abs(got - e_ref) <= 1e-12 * max(1.0, abs(e_ref)) and abs(norm - n_ref) <= 1e-12 * n_ref
        else:
            assert energy_error(got, e_ref, terms, n) <= 4e-7 and abs(norm - n_ref) <= 1e-6 * n_ref
