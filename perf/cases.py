"""Workloads the engine is timed on: one pass each through its public entry points.

The kinds follow the engine's workload families and its device-pointer
primitives, at the sizes of the bundled configurations (bench, tests) or of
the same shape:

  sweep     variational sweep: shared hardware-efficient prefix, one suffix
            and one Pauli-sum energy per task, executed from its plan
  noisy     noisy multishot trajectories: plan execution, samples
  qec       rotated-surface-code memory: plan execution, syndrome bits
  clifford  stabilizer tasks with random measurement outcomes
  mixed     independent random-circuit groups of several register sizes
  apply     a gate list on the caller's device state
  energy    Pauli-sum energy of the caller's device state
  sample    shots from the caller's device state
  dense     fused dense blocks on the caller's device state
  train     one training step of the cost model (loss, gradient, Adam)

Energies of FP32-mode tasks are handed on in FP32, the type of the states
they are taken of; those of FP64-mode tasks in FP64.
"""
import math

import numpy as np
import torch

from paper_2609_23664_gb300 import quwarp as Q
from paper_2609_23664_gb300 import workloads as W

_engine = None


def engine():
    """One engine per process, as a program keeps it (it holds the tile tuning)."""
    global _engine
    if _engine is None:
        _engine = Q.Engine(0)
    return _engine


def listed():
    return [
        # the smallest calls: one optimizer step of the cost model on a batch
        # of measured timings (latency and launches)
        {"name": "train_256", "kind": "train", "batch": 256},
        # the plain 12-qubit sweep in complex128: small states, many kernels
        # per microsecond of work
        {"name": "sweep12_fp64", "kind": "sweep", "n": 12, "fp64": True, "layers": 6, "tasks": 16, "max_layers": 1,
         "terms": 20},
        # an ordinary sweep, states that stay in L2
        {"name": "sweep20", "kind": "sweep", "n": 20, "fp64": False, "layers": 20, "tasks": 64, "max_layers": 4,
         "terms": 200},
        # the batched 24-qubit sweep, states larger than L2 (a quarter of the
        # full sweep's tasks)
        {"name": "sweep24", "kind": "sweep", "n": 24, "fp64": False, "layers": 20, "tasks": 64, "max_layers": 4,
         "terms": 200},
        # noisy multishot study at 22 qubits
        {"name": "noisy22", "kind": "noisy", "n": 22, "gates": 400, "traj": 1024, "shots": 100},
        # surface-code memory d=15, Pauli errors in the last rounds
        {"name": "qec15", "kind": "qec", "d": 15, "shared": 100, "rounds": 5, "tasks": 4096},
        # stabilizer circuits with random outcomes: every task on its own tableau
        {"name": "clifford100", "kind": "clifford", "n": 100, "depth": 40, "own_depth": 10, "tasks": 256},
        # groups of random circuits at several register sizes, own energies
        {"name": "mixed", "kind": "mixed", "n_min": 16, "n_max": 22, "tasks": 40, "terms": 8},
        # device-pointer primitives, one call each
        {"name": "apply24", "kind": "apply", "n": 24, "fp64": False, "gates": 200},
        {"name": "energy26", "kind": "energy", "n": 26, "fp64": False, "terms": 100},
        {"name": "sample26", "kind": "sample", "n": 26, "fp64": False, "shots": 4096},
        {"name": "dense26", "kind": "dense", "n": 26, "layers": 2},
    ]


def draw(rng):
    def lg(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["train", "sweep", "sweep", "noisy", "qec", "clifford", "mixed", "apply", "energy", "sample",
                       "dense"])
    if kind == "train":
        return {"kind": kind, "batch": lg(1, 4096)}
    if kind == "sweep":
        fp64 = rng.random() < 0.25
        return {"kind": kind, "n": rng.randint(6, 14) if fp64 else rng.randint(8, 22), "fp64": fp64,
                "layers": lg(2, 20), "tasks": lg(2, 64), "max_layers": rng.randint(1, 4), "terms": lg(4, 200)}
    if kind == "noisy":
        return {"kind": kind, "n": rng.randint(8, 21), "gates": lg(40, 400), "traj": lg(16, 512), "shots": lg(1, 200)}
    if kind == "qec":
        return {"kind": kind, "d": rng.choice([3, 5, 7, 9, 11, 13, 15]), "shared": lg(3, 100), "rounds": rng.randint(1, 5),
                "tasks": lg(16, 4096)}
    if kind == "clifford":
        return {"kind": kind, "n": lg(5, 150), "depth": lg(4, 40), "own_depth": lg(1, 12), "tasks": lg(4, 256)}
    if kind == "mixed":
        lo = rng.randint(8, 18)
        return {"kind": kind, "n_min": lo, "n_max": rng.randint(lo, 20), "tasks": lg(6, 40), "terms": lg(2, 16)}
    if kind == "apply":
        fp64 = rng.random() < 0.3
        return {"kind": kind, "n": rng.randint(5, 21) if fp64 else rng.randint(5, 24), "fp64": fp64, "gates": lg(5, 300)}
    if kind == "energy":
        fp64 = rng.random() < 0.3
        return {"kind": kind, "n": rng.randint(5, 20) if fp64 else rng.randint(5, 26), "fp64": fp64, "terms": lg(1, 200)}
    if kind == "sample":
        fp64 = rng.random() < 0.3
        return {"kind": kind, "n": rng.randint(5, 24) if fp64 else rng.randint(5, 26), "fp64": fp64, "shots": lg(1, 8192)}
    return {"kind": kind, "n": rng.randint(12, 26), "layers": rng.randint(1, 3)}


# ---- inputs ------------------------------------------------------------------------

def _rng(case, seed):
    return np.random.default_rng([20260923, seed])


def _state(n, fp64, seed):
    """A random normalized state (the shape of a deep circuit's output)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    v = torch.randn((1 << n, 2), generator=g, device="cuda", dtype=torch.float64 if fp64 else torch.float32)
    v /= torch.linalg.vector_norm(v)
    return torch.view_as_complex(v)


def _sweep_tasks(case, seed):
    mode = W.MODE_SV_FP64 if case["fp64"] else W.MODE_SV_FP32
    return W.vqe24_sweep(seed=seed, n=case["n"], prefix_layers=case["layers"], n_tasks=case["tasks"],
                         max_suffix_layers=case["max_layers"], n_terms=case["terms"], mode=mode)


def _qec_tasks(case, seed):
    """The surface-code memory of workloads.qec_surface_code_tasks (its error
    draws taken at once)."""
    rng = _rng(case, seed)
    code = W.rotated_surface_code(case["d"])
    prefix = W.concat(*[W.syndrome_round(code, rng) for _ in range(case["shared"])])
    cycle = W.syndrome_round(code, rng)
    hit = rng.random((case["tasks"], case["rounds"], code.n_data, 2)) < 1e-3
    tasks = []
    for t in range(case["tasks"]):
        spans = [prefix]
        for r in range(case["rounds"]):
            err = [(W.OP_Z if k else W.OP_X, int(q), 0) for q, k in zip(*np.nonzero(hit[t, r]))]
            if err:
                spans.append(W.gates_from_list(err))
            spans.append(cycle)
        tasks.append(W.Task(mode=W.MODE_TABLEAU, n=code.n, spans=spans))
    return tasks


def _clifford_tasks(case, seed):
    rng = _rng(case, seed)
    n = case["n"]
    prefix = W.random_clifford_layers(rng, n, case["depth"])
    tasks = []
    for _ in range(case["tasks"]):
        own = W.random_clifford_layers(rng, n, case["own_depth"])
        meas = W.gates_from_list([(W.OP_MEASURE, q, 0, float(rng.integers(0, 2))) for q in range(n)])
        tasks.append(W.Task(mode=W.MODE_TABLEAU, n=n, spans=[prefix, own, meas]))
    return tasks


def _mixed_tasks(case, seed):
    return W.mixed_planned(seed=seed, n_tasks=case["tasks"], n_min=case["n_min"], n_max=case["n_max"], group_max=12,
                           n_terms=case["terms"])


def _tasks(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        return _sweep_tasks(case, seed)
    if kind == "noisy":
        return W.noisy22_trajectories(seed=seed, n=case["n"], n_gates=case["gates"], n_traj=case["traj"],
                                      shots=case["shots"])
    if kind == "qec":
        return _qec_tasks(case, seed)
    if kind == "clifford":
        return _clifford_tasks(case, seed)
    return _mixed_tasks(case, seed)


def _mlp_inputs(case, seed):
    """Normalized features, log2-ns targets and He-initialized parameters."""
    rng = _rng(case, seed)
    x = rng.normal(size=(case["batch"], Q.MLP_IN)).astype(np.float32)
    t = (16 + 3 * rng.normal(size=case["batch"])).astype(np.float32)
    i, h = Q.MLP_IN, Q.MLP_HID
    p = np.zeros(Q.MLP_PARAMS, np.float32)
    at = 0
    for count, fan in ((i * h, i), (h, 0), (h * h, h), (h, 0), (h, h), (1, 0)):
        if fan:
            a = math.sqrt(6.0 / fan)
            p[at:at + count] = rng.uniform(-a, a, count)
        at += count
    p[-1] = t.mean()
    return p, x, t


def _dense_gates(case, seed):
    return W.hea_circuit(_rng(case, seed), case["n"], case["layers"])


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("sweep", "noisy", "qec", "clifford", "mixed"):
        tasks = _tasks(case, seed)
        # shots are reproducible from run to run only for a fixed tile shape
        # (plain FP32 rounding follows it)
        opts = {"tile_qubits": 13, "low_qubits": 4} if kind == "noisy" else {}
        wl = Q.Workload(tasks)
        plan = Q.Plan(engine(), wl, **opts)
        return {"kind": kind, "tasks": tasks, "wl": wl, "plan": plan, "fp64": case.get("fp64", False)}
    if kind == "train":
        p, x, t = (torch.from_numpy(a).cuda() for a in _mlp_inputs(case, seed))
        z = torch.zeros_like
        return {"kind": kind, "p": p, "x": x, "t": t, "m": z(p), "v": z(p), "g": z(p), "batch": case["batch"],
                "loss": torch.zeros(1, device="cuda"), "step": 0}
    n, fp64 = case["n"], case.get("fp64", False)
    s = {"kind": kind, "n": n, "fp64": fp64, "mode": W.MODE_SV_FP64 if fp64 else W.MODE_SV_FP32,
         "state": _state(n, fp64, seed)}
    rng = _rng(case, seed)
    if kind == "apply":
        s["gates"] = W.random_circuit(rng, n, case["gates"])
    elif kind == "energy":
        s["terms"] = W.random_pauli_hamiltonian(rng, n, case["terms"])
    elif kind == "sample":
        s["uniforms"] = rng.random(case["shots"])
    else:
        s["prog"] = Q.DenseProgram(engine(), s["mode"], n, _dense_gates(case, seed))
    engine()
    return s


def run(s):
    kind = s["kind"]
    if kind in ("sweep", "mixed"):
        plan = s["plan"].run()
        en = np.array([plan.energy(t) for t in range(len(s["tasks"]))])
        en = en if s["fp64"] else en.astype(np.float32)
        return {"energy": en[:, 0], "norm": en[:, 1]}
    if kind == "noisy":
        plan = s["plan"].run()
        return np.concatenate([plan.samples(t) for t in range(len(s["tasks"]))]).astype(np.int64)
    if kind in ("qec", "clifford"):
        plan = s["plan"].run()
        return np.concatenate([plan.syndrome(t) for t in range(len(s["tasks"]))])
    if kind == "train":
        s["step"] += 1
        Q.mlp_loss_grad_dev(s["p"].data_ptr(), s["x"].data_ptr(), s["t"].data_ptr(), s["batch"],
                            s["loss"].data_ptr(), s["g"].data_ptr())
        Q.mlp_adam_dev(s["p"].data_ptr(), s["g"].data_ptr(), s["m"].data_ptr(), s["v"].data_ptr(), Q.MLP_PARAMS,
                       s["step"])
        return {"loss": s["loss"], "grad": s["g"], "params": s["p"]}
    st = s["state"].data_ptr()
    if kind == "apply":
        Q.sv_apply_dev(engine(), s["mode"], s["n"], st, s["gates"])
        return s["state"]
    if kind == "energy":
        en = np.array(Q.sv_energy_dev(engine(), s["mode"], s["n"], st, s["terms"]))
        return en if s["fp64"] else en.astype(np.float32)
    if kind == "sample":
        return Q.sv_sample_dev(engine(), s["mode"], s["n"], st, s["uniforms"]).astype(np.int64)
    s["prog"].run(st)
    return s["state"]


# ---- what a pass cannot do without ---------------------------------------------------

def _gate_flops(g):
    """Real operations per amplitude of a gate list: 7 for a rotation or H
    (two complex-by-real products and an add, rounded up), 6 for half the
    amplitudes of a phase, none for a permutation or a sign."""
    op = g["op"]
    return float(7 * np.isin(op, (W.OP_H, W.OP_RX, W.OP_RY)).sum() + 3 * np.isin(op, (W.OP_RZ, W.OP_PHASE)).sum())


def work(case):
    kind = case["kind"]
    if kind == "train":
        b, n = case["batch"], Q.MLP_PARAMS
        return {"bytes": 4 * (13 * b + 8 * n), "flops": 6 * b * n + 12 * n}
    if kind in ("sweep", "noisy", "mixed"):
        # every boundary and final state made once; gate arithmetic of the
        # shared prefix once and of each suffix; 4 operations per amplitude
        # and Pauli term; sampling reads its state once
        if kind == "sweep":
            n, amp = case["n"], (16 if case["fp64"] else 8)
            dim, layer = float(2 ** case["n"]), 10.0 * case["n"]
            suf = case["tasks"] * (1 + case["max_layers"]) / 2
            return {"bytes": amp * dim * (1 + case["tasks"]),
                    "flops": dim * (layer * (case["layers"] + suf) + 4.0 * case["terms"] * case["tasks"])}
        if kind == "noisy":
            dim = float(2 ** case["n"])
            errors = 1.0 - math.exp(-1e-3 * case["gates"])  # share of trajectories with an error
            states = 1 + errors * case["traj"]
            return {"bytes": 8 * dim * states, "flops": dim * states * case["gates"] * 0.5 * 3.4}
        dim = sum(2.0 ** n for n in range(case["n_min"], case["n_max"] + 1)) / (case["n_max"] - case["n_min"] + 1)
        return {"bytes": 8 * dim * case["tasks"], "flops": dim * case["tasks"] * (150 * 3.4 + 4.0 * case["terms"])}
    if kind in ("qec", "clifford"):
        # tableau rows (x and z bits) read and written once; two row words per
        # gate and 64 qubits
        n = 2 * case["d"] ** 2 - 1 if kind == "qec" else case["n"]
        if kind == "qec":
            meas = n // 2 * (case["shared"] + case["rounds"] * case["tasks"])
            return {"bytes": 2 * n * n / 2 + meas, "flops": 4.0 * n * n / 64 * case["shared"] * 4}
        return {"bytes": case["tasks"] * (n * n + n),
                "flops": 4.0 * n * n / 64 * (case["depth"] + case["tasks"] * (case["own_depth"] + n))}
    amp = 16 if case.get("fp64") else 8
    dim = float(2 ** case["n"])
    if kind == "apply":
        return {"bytes": 2 * amp * dim, "flops": dim * case["gates"] * 3.4}
    if kind == "energy":
        return {"bytes": amp * dim, "flops": dim * (4.0 * case["terms"] + 4)}
    if kind == "sample":
        return {"bytes": amp * dim, "flops": 4 * dim}
    blocks = case["layers"] * math.ceil((case["n"] - 1) / 4)
    return {"bytes": 2 * amp * dim, "flops": blocks * dim * 32 * 8.0}


# ---- the same results in 64 bits -------------------------------------------------------

def _mat(g):
    op, th = int(g["op"]), float(g["theta"])
    c, s = math.cos(th / 2), math.sin(th / 2)
    r = math.sqrt(0.5)
    e = complex(c, s)
    return {W.OP_H: [[r, r], [r, -r]], W.OP_X: [[0, 1], [1, 0]], W.OP_Y: [[0, -1j], [1j, 0]],
            W.OP_Z: [[1, 0], [0, -1]], W.OP_RX: [[c, -1j * s], [-1j * s, c]], W.OP_RY: [[c, -s], [s, c]],
            W.OP_RZ: [[e.conjugate(), 0], [0, e]]}[op]


def _evolve(psi, n, gates):
    """Gates on a complex128 state; neighbouring one-qubit gates of a qubit
    are multiplied first, runs of CNOTs become one index permutation."""
    dev = psi.device
    pend, perm = {}, None

    def flush(q):
        nonlocal psi
        m = pend.pop(q, None)
        if m is None:
            return
        v = psi.view(-1, 2, 1 << q)
        a, b = v[:, 0], v[:, 1]
        (u00, u01), (u10, u11) = m.tolist()
        out = torch.empty_like(v)
        if u01 == 0 and u10 == 0:
            out[:, 0], out[:, 1] = a * u00, b * u11
        else:
            out[:, 0], out[:, 1] = a * u00 + b * u01, a * u10 + b * u11
        psi = out.view(-1)

    def flush_perm():
        nonlocal psi, perm
        if perm is not None:
            psi = psi[perm]
            perm = None

    x = None
    for g in gates:
        op, q0, q1 = int(g["op"]), int(g["q0"]), int(g["q1"])
        if op == W.OP_CNOT:
            flush(q0)
            flush(q1)
            if x is None:
                x = torch.arange(1 << n, device=dev)
            # new[y] = old[cnot(y)]; a later CNOT acts on the index first
            step = x ^ (((x >> q0) & 1) << q1)
            perm = step if perm is None else perm[step]
        elif op == W.OP_CZ:
            flush_perm()
            flush(q0)
            flush(q1)
            hi, lo = max(q0, q1), min(q0, q1)
            psi = psi.clone()
            psi.view(-1, 2, 1 << (hi - lo - 1), 2, 1 << lo)[:, 1, :, 1] *= -1
        else:
            flush_perm()
            m = np.array(_mat(g), dtype=complex)
            pend[q0] = m @ pend[q0] if q0 in pend else m
    flush_perm()
    for q in list(pend):
        flush(q)
    return psi


def _energies(psi, n, terms):
    """sum_k c_k <P_k> / <psi|psi> and <psi|psi>, P|x> = i^{#Y}(-1)^{popc(x & z)}|x ^ m>."""
    dev = psi.device
    lo_n = n // 2
    hi_n = n - lo_n
    v = psi.view(1 << hi_n, 1 << lo_n)
    lo, hi = torch.arange(1 << lo_n, device=dev), torch.arange(1 << hi_n, device=dev)

    par = hi.clone()
    for sh in (8, 4, 2, 1):
        par ^= par >> sh
    flip = (1 - 2 * (par & 1)).double()  # (-1)^popc(x), x < 2^hi_n

    norm = float(psi.abs().square().sum())
    total = torch.zeros((), dtype=torch.float64, device=dev)
    for t in terms:
        m, z, c = int(t["xmask"]), int(t["zmask"]), float(t["coef"])
        mm, zl, zh = (1 << lo_n) - 1, z & ((1 << lo_n) - 1), z >> lo_n
        ys = bin(m & z).count("1")
        p = v[hi ^ (m >> lo_n)][:, lo ^ (m & mm)] if m else v
        # <psi|P|psi> = sum_x conj(psi[x ^ m]) i^ys (-1)^{x.z} psi[x]
        f = p.real * v.imag - p.imag * v.real if ys & 1 else p.real * v.real + p.imag * v.imag
        e = flip[hi & zh] @ (f @ flip[lo & zl])
        total += c * (1, -1, -1, 1)[ys & 3] * e
    return float(total) / norm, norm


def _exact_tasks(tasks):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    prefixes, out = {}, []
    count = {}
    for t in tasks:
        count[id(t.spans[0])] = count.get(id(t.spans[0]), 0) + 1
    for t in tasks:
        key = (id(t.spans[0]), t.n)
        if key not in prefixes:
            psi = torch.zeros(1 << t.n, dtype=torch.complex128, device=dev)
            psi[0] = 1
            psi = _evolve(psi, t.n, t.spans[0])
            if count[id(t.spans[0])] > 1:
                prefixes.clear()
                prefixes[key] = psi
        else:
            psi = prefixes[key]
        rest = t.spans[1:]
        if rest:
            psi = _evolve(psi, t.n, np.concatenate(rest))
        out.append(_energies(psi, t.n, t.terms))
    out = np.array(out)
    return {"energy": out[:, 0], "norm": out[:, 1]}


def _exact_train(case, seed):
    """Loss, gradient and one Adam step in 64 bits, on the BF16-rounded
    weights, inputs and activations the network is defined with."""
    p32, x32, t32 = (torch.from_numpy(a) for a in _mlp_inputs(case, seed))

    def bf(a):
        return a.float().bfloat16().double()

    i, h = Q.MLP_IN, Q.MLP_HID
    w1, b1, w2, b2, w3, b3 = torch.split(bf(p32), [i * h, h, h * h, h, h, 1])
    w1, w2 = w1.view(h, i), w2.view(h, h)
    x, t = bf(x32), t32.double()
    a1 = x @ w1.T + b1
    h1 = bf(a1.clamp_min(0))
    a2 = h1 @ w2.T + b2
    h2 = bf(a2.clamp_min(0))
    d = h2 @ w3 + b3 - t
    dy = 2 * d / len(t)
    da2 = dy[:, None] * w3 * (a2 > 0)
    da1 = (da2 @ w2) * (a1 > 0)
    g = torch.cat([(da1.T @ x).reshape(-1), da1.sum(0), (da2.T @ h1).reshape(-1), da2.sum(0), h2.T @ dy,
                   dy.sum()[None]])
    # the first Adam step: both moments corrected for their start at zero
    params = p32.double() - 1e-3 * g / (g.abs() + 1e-8)
    return {"loss": d.square().mean().reshape(1), "grad": g, "params": params}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("noisy", "qec", "clifford", "sample"):
        return None  # whole numbers
    if kind == "train":
        return _exact_train(case, seed)
    if kind in ("sweep", "mixed"):
        return _exact_tasks(_tasks(case, seed))
    n = case["n"]
    psi = _state(n, case.get("fp64", False), seed).to(torch.complex128)
    rng = _rng(case, seed)
    if kind == "apply":
        return _evolve(psi, n, W.random_circuit(rng, n, case["gates"]))
    if kind == "energy":
        return np.array(_energies(psi, n, W.random_pauli_hamiltonian(rng, n, case["terms"])))
    return _evolve(psi, n, _dense_gates(case, seed))
