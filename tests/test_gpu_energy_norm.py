"""Norms of FP32 states, which every energy is divided by: states of constant
amplitude, whose rounding is the same in every sum, at the sizes where a thread
takes one, four and sixteen runs of representatives.

Tolerance: a square rounds once and a pair of squares once more, together
1.5 x 2^-24 of the pair; sums of equal numbers in a tree are exact, and adding
real and imaginary parts rounds once: 2.5 x 2^-24.  Beyond 2^-24 of that the
sums are kept in pairs."""
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


@pytest.mark.parametrize("n,offset", [(5, 0), (8, 0), (8, 1), (16, 0), (16, 1), (24, 0), (26, 0), (28, 0)])
@pytest.mark.parametrize("re,im", [(1.3733253479003906, 0.0), (1.0002427101135254, 0.0), (1.4868028163909912, 1.054221749305725)])
def test_norm_of_a_constant_state(eng, n, offset, re, im):
    # offset 1: a state off the 16-byte boundary
    st = torch.full(((1 << n) + offset,), complex(re, im), dtype=torch.complex64, device="cuda")[offset:]
    terms = W.random_pauli_hamiltonian(np.random.default_rng(n), n, 3)
    _, norm = Q.sv_energy_dev(eng, W.MODE_SV_FP32, n, st.data_ptr(), terms)
    r, i = float(np.float32(re)), float(np.float32(im))
    assert abs(norm / ((r * r + i * i) * 2.0 ** n) - 1) <= 2.5 * 2.0 ** -24
