"""Gradient workspace of the cost model, on the host: training allocates it
once for its batch size and reuses it for the shorter last batch of an epoch,
so the workspace of a batch has to cover the CTAs of every smaller one."""
import ctypes

import numpy as np
import pytest

from paper_2609_23664_gb300 import quwarp as Q

N_PARTIAL = Q.MLP_PARAMS + 1  # floats of one CTA: the gradient and the loss


def _fn(name, res):
    f = getattr(Q.lib(), name)  # C++ functions of the library, by their mangled names
    f.restype, f.argtypes = res, [ctypes.c_uint32]
    return f


def test_workspace_covers_every_shorter_batch():
    scratch = _fn("_ZN2qw18mlp_scratch_floatsEj", ctypes.c_size_t)
    have = np.array([scratch(b) for b in range(1, 8001)], dtype=np.int64)
    assert np.all(have[:-1] <= have[1:])


@pytest.mark.parametrize("batch", [1, 99, 100, 101, 200, 256, 1024, 3200, 3201, 65536, 1 << 20])
def test_ctas_fit_the_workspace(batch):
    scratch = _fn("_ZN2qw18mlp_scratch_floatsEj", ctypes.c_size_t)
    ctas = _fn("_ZN2qw13mlp_grad_ctasEj", ctypes.c_uint32)
    have = scratch(batch)
    for b in range(max(1, batch - 4000), batch + 1):
        assert ctas(b) * N_PARTIAL <= have, b


@pytest.mark.parametrize("batch", [1, 31, 100, 3199, 3200, 3201, 6400, 65536, 65537, 1 << 24, (1 << 32) - 1])
def test_no_cta_takes_more_than_32_samples(batch):
    # samples of a CTA run one after another, in gradients and in forward passes
    ctas = _fn("_ZN2qw13mlp_grad_ctasEj", ctypes.c_uint32)(batch)
    assert batch <= 32 * ctas and ctas <= batch
