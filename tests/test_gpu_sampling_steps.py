"""Shots whose target falls next to empty blocks, to the last bit.

The offsets of a state's blocks come from a scan, whose sums round in another
order at each end of an empty block; a target in such a step of one ulp must
still give an outcome beside it, not one elsewhere in the state.  The scan is
replayed here in FP64 (runs of blocks by 256 threads, a warp scan of the runs'
sums, the warps in order) to find the steps; each nonempty block holds one
outcome, so the block sums are known exactly.

Tolerance: an outcome is beside its target when its interval of the exact
distribution comes within 1e-12 of it (256 sums of FP64)."""
import numpy as np
import pytest

from paper_2609_23664_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2609_23664_gb300 import quwarp as Q  # noqa: E402


def _scan(bsum):
    n, run = len(bsum), -(-len(bsum) // 256)
    acc = np.zeros(256)
    for k in range(run):
        b = np.arange(256) * run + k
        acc = acc + np.where(b < n, bsum[np.minimum(b, n - 1)], 0.0)
    incl = acc.reshape(8, 32).copy()
    for d in (1, 2, 4, 8, 16):
        up = incl.copy()
        incl[:, d:] = incl[:, d:] + up[:, :-d]
    before = np.zeros(8)
    for w in range(1, 8):
        before[w] = before[w - 1] + incl[w - 1, 31]
    excl = np.concatenate([np.zeros((8, 1)), incl[:, :-1]], axis=1)
    base = (before[:, None] + excl).reshape(256)
    o = np.zeros(n + 1)
    for k in range(run):
        b = np.arange(256) * run + k
        m = b < n
        o[b[m]] = base[m]
        base = base + np.where(m, bsum[np.minimum(b, n - 1)], 0.0)
    o[n] = before[7] + incl[7, 31]
    return o


@pytest.mark.parametrize("n,fill", [(20, 0.5), (20, 0.05), (21, 0.5), (22, 0.3), (22, 0.01), (24, 0.4), (16, 0.5)])
def test_targets_in_the_steps_of_empty_blocks(n, fill):
    rng = np.random.default_rng(n)
    nb = 1 << (n - 12)
    full = rng.random(nb) < fill
    full[rng.integers(0, nb)] = True
    amp = np.where(full, rng.uniform(0.1, 1.0, nb), 0.0)
    psi = np.zeros(1 << n, dtype=np.complex128)
    psi[(np.arange(nb) << 12) + rng.integers(0, 4096, nb)] = amp
    p = amp * amp
    o = _scan(p)
    total = o[nb]
    u = []
    for b in np.nonzero(~full & (o[1:] > o[:-1]))[0]:
        for k in range(-2, 3):  # a uniform whose target lies in the step
            v = o[b] / total
            for _ in range(abs(k)):
                v = np.nextafter(v, 2.0 if k > 0 else -1.0)
            if o[b] <= v * total < o[b + 1] and 0.0 <= v < 1.0:
                u.append(v)
                break
    print("n %d: %d steps hit" % (n, len(u)))
    u = np.array(u + list(rng.random(200)) + [0.0, np.nextafter(1.0, 0.0)])
    eng = Q.Engine(0)
    st = torch.tensor(psi, device="cuda")
    got = Q.sv_sample_dev(eng, W.MODE_SV_FP64, n, st.data_ptr(), u).astype(np.int64)
    eng.close()
    pp = np.abs(psi) ** 2
    assert np.all(pp[got] > 0)
    cdf = np.cumsum(pp) / pp.sum()
    lo = np.where(got > 0, cdf[got - 1], 0.0)
    assert np.all((u >= lo - 1e-12) & (u <= cdf[got] + 1e-12))
