"""The work a user of this framework has it do, as measurable cases through its public calls.

A case is a dict of plain values; ``kind`` says which entry points it goes through:

* ``circuit``      one noisy circuit on a ``Density`` (plain or fused mode), with the readouts a noise
                   study takes and the final matrix in the caller's own device tensor
* ``wide``         the wider operations: controlled gates, dense gates on 2 to 5 qubits, a 3-qubit channel
* ``experiment``   the paper's multi-qubit noise experiment, density form: every step one channel on the
                   whole register, then a gate of the algorithm, then readouts
* ``multiverse``   the statevector form: noise steps on many trajectories, gates, the density matrix
* ``observables``  every readout on a given state, then a measurement
* ``batch``        independent circuits of uneven size in one launch
* ``serve``        a queue of requests through the serving loop

The state is held and evolved in complex64, so readouts are returned as float32 / complex64.
"""

from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1101_1785_gb300 as q

C128 = np.complex128
_SQ2 = 1.0 / math.sqrt(2.0)
ONE = {
    "H": np.array([[_SQ2, _SQ2], [_SQ2, -_SQ2]], C128),
    "X": np.array([[0, 1], [1, 0]], C128),
    "Y": np.array([[0, -1j], [1j, 0]], C128),
    "Z": np.array([[1, 0], [0, -1]], C128),
    "S": np.array([[1, 0], [0, 1j]], C128),
    "T": np.array([[1, 0], [0, np.exp(0.25j * np.pi)]], C128),
}
CNOT = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, 0, 1], [0, 0, 1, 0]], C128)
CZ = np.diag([1, 1, 1, -1]).astype(C128)


def listed():
    return [
        # the paper's own scale: a 4-qubit noisy circuit, one launch per operation, measured at the end
        {"name": "plain_n4", "kind": "circuit", "n": 4, "gates": 40, "mix": "mixed", "noise": "adpd", "fused": False,
         "init": "zero", "chunk": 0},
        # the paper's five-qubit noise study (GHZ chain, 17-term channel on the register every step)
        {"name": "experiment_n5", "kind": "experiment", "n": 5, "steps": 8, "paths": 8},
        # the same study as sampled trajectories
        {"name": "multiverse_n5", "kind": "multiverse", "n": 5, "vectors": 2048, "steps": 8, "densities": 8},
        # a one-off circuit of ordinary size in fused mode
        {"name": "fused_n9", "kind": "circuit", "n": 9, "gates": 200, "mix": "mixed", "noise": "adpd", "fused": True,
         "init": "zero", "chunk": 0},
        # the 12-qubit depolarising circuit, one launch per gate and per channel
        {"name": "plain_n12", "kind": "circuit", "n": 12, "gates": 30, "mix": "haar70", "noise": "dep", "fused": False,
         "init": "matrix", "chunk": 0},
        # controlled, dense two- to five-qubit gates and a three-qubit channel
        {"name": "wide_n12", "kind": "wide", "n": 12, "rounds": 1},
        # readouts of a 13-qubit state, as taken between the steps of a noise study
        {"name": "observables_n13", "kind": "observables", "n": 13, "keep": 6},
        # trajectories at a size where forming the density matrix is the work
        {"name": "multiverse_n13", "kind": "multiverse", "n": 13, "vectors": 64, "steps": 2, "densities": 1},
        # the 14-qubit noisy circuit in fused mode with a checkpoint every 100 gates
        {"name": "fused_n14", "kind": "circuit", "n": 14, "gates": 200, "mix": "mixed", "noise": "adpd", "fused": True,
         "init": "zero", "chunk": 100},
        # the largest register whose states fit the card several times over
        {"name": "fused_n15", "kind": "circuit", "n": 15, "gates": 60, "mix": "haar70", "noise": "dep", "fused": True,
         "init": "zero", "chunk": 0},
        # circuits of 4 to 10 qubits, 50 to 400 gates deep, in one captured launch
        {"name": "batch_64", "kind": "batch", "circuits": 64, "nmin": 4, "nmax": 10, "dmin": 50, "dmax": 400},
        # a burst of serving requests, small ones most often
        {"name": "serve_48", "kind": "serve", "requests": 48, "nmin": 3, "nmax": 11, "dmin": 20, "dmax": 300},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["circuit", "circuit", "circuit", "circuit", "wide", "experiment", "multiverse", "observables",
                       "batch", "serve"])
    if kind == "circuit":
        fused = rng.random() < 0.65
        n = rng.randint(3, 15 if fused else 13)
        gates = _log_int(rng, 20, 60 if n == 15 else 200 if n >= 13 else 400) if fused else _log_int(rng, 5, 60 if n < 13 else 12)
        init = "matrix" if n <= 12 and rng.random() < 0.4 else "zero"
        return {"kind": kind, "n": n, "gates": gates, "mix": rng.choice(["mixed", "haar70"]),
                "noise": rng.choice(["adpd", "adpd", "dep", "none"]), "fused": fused, "init": init,
                "chunk": rng.choice([0, 50, 100])}
    if kind == "wide":
        n = rng.randint(6, 13)
        return {"kind": kind, "n": n, "rounds": 1 if n >= 11 else rng.randint(1, 3)}
    if kind == "experiment":
        return {"kind": kind, "n": rng.randint(2, 5), "steps": _log_int(rng, 4, 40), "paths": rng.randint(2, 15)}
    if kind == "multiverse":
        n = rng.randint(3, 13)
        vectors = _log_int(rng, 8, min(4096, 1 << (20 - n)) if n < 12 else 96)
        return {"kind": kind, "n": n, "vectors": vectors, "steps": rng.randint(1, 10),
                "densities": rng.randint(1, 8) if n < 10 else 1}
    if kind == "observables":
        n = rng.randint(4, 13)
        return {"kind": kind, "n": n, "keep": rng.randint(2, min(6, n - 1))}
    if kind == "batch":
        nmin = rng.randint(3, 6)
        nmax = rng.randint(max(nmin + 1, 7), 10)
        dmin = _log_int(rng, 20, 100)
        return {"kind": kind, "circuits": _log_int(rng, 8, 64), "nmin": nmin, "nmax": nmax, "dmin": dmin,
                "dmax": dmin + _log_int(rng, 20, 300)}
    nmin = rng.randint(3, 5)
    dmin = _log_int(rng, 20, 60)
    return {"kind": kind, "requests": _log_int(rng, 4, 48), "nmin": nmin, "nmax": rng.randint(nmin + 2, 11),
            "dmin": dmin, "dmax": dmin + _log_int(rng, 20, 240)}


# ----------------------------------------------------------------------------- inputs


class Op:
    """A gate (one matrix) or channel (Kraus operators) on qubits, as PackedOps and Density.apply_op take it."""

    def __init__(self, kind, qubits, mats):
        self.kind, self.qubits, self.mats = kind, tuple(int(x) for x in qubits), np.asarray(mats, C128)

    @property
    def k(self):
        return len(self.qubits)


class Circuit:
    def __init__(self, n, ops):
        self.n, self.ops = n, ops


def _su2(rng):
    a, b, c, d = rng.standard_normal(4)
    s = 1.0 / math.sqrt(a * a + b * b + c * c + d * d)
    return np.array([[a + 1j * b, c + 1j * d], [-c + 1j * d, a - 1j * b]]) * s


def _unitary(rng, d):
    z = rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d))
    u, r = np.linalg.qr(z)
    return u * (np.diag(r) / np.abs(np.diag(r)))[None, :]


def _channels(noise, gamma):
    if noise == "adpd":
        lam = 0.02
        return [np.array([[[1, 0], [0, math.sqrt(1 - gamma)]], [[0, math.sqrt(gamma)], [0, 0]]], C128),
                np.array([[[1, 0], [0, math.sqrt(1 - lam)]], [[0, 0], [0, math.sqrt(lam)]]], C128)]
    if noise == "dep":
        p = 1e-3
        return [np.stack([math.sqrt(1 - p) * np.eye(2), *(math.sqrt(p / 3) * ONE[x] for x in "XYZ")]).astype(C128)]
    return []


def _circuit_ops(rng, n, gates, mix, noise, gamma=0.01):
    """Gates drawn as in the framework's workloads ("mixed": H, X, Z, S, T, CNOT, Haar alike; "haar70": 70 % Haar,
    the rest CNOT or CZ), each followed by the noise channels on the qubits it touched."""
    ch = _channels(noise, gamma)
    out = []
    for _ in range(gates):
        if mix == "mixed":
            name = ("H", "X", "Z", "S", "T", "CNOT", "HAAR")[int(rng.integers(7))]
        else:
            name = "HAAR" if rng.random() < 0.7 else ("CNOT", "CZ")[int(rng.integers(2))]
        if name in ("CNOT", "CZ"):
            qs = tuple(int(x) for x in rng.choice(n, size=2, replace=False))
            out.append(Op("gate", qs, (CNOT if name == "CNOT" else CZ)[None]))
        else:
            qs = (int(rng.integers(n)),)
            out.append(Op("gate", qs, (_su2(rng) if name == "HAAR" else ONE[name])[None]))
        for x in qs:
            out.extend(Op("kraus", (x,), k) for k in ch)
    return out


def _density_matrix(n, seed, rank=4, mixed=0.5):
    """mixed * 1 / 2^n + (1 - mixed) * a random state of the given rank, exactly Hermitian, on the GPU (complex64)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    a = torch.randn(1 << n, rank, dtype=torch.complex64, device="cuda", generator=g)
    a /= torch.linalg.vector_norm(a)
    rho = a @ a.conj().T
    rho = (rho + rho.conj().T) * (0.5 * (1 - mixed))
    rho.diagonal().add_(mixed / (1 << n))
    return rho.contiguous()


def _wide_ops(rng, n, rounds):
    """(call, arguments) of one round: what circuits with wider operations than CNOT contain."""
    out = []
    for _ in range(rounds):
        p = [int(x) for x in rng.permutation(n)]
        out.append(("gate1", ONE["X"], (p[2],), (p[0], p[1])))  # Toffoli
        out.append(("gate1", _su2(rng), (p[3],), (p[4],)))  # controlled one-qubit gate
        out.append(("gate2", _unitary(rng, 4), (p[1], p[3]), (p[5],)))  # controlled two-qubit gate
        out.append(("gate2", _unitary(rng, 4), (p[0], p[2]), ()))  # general two-qubit gate
        ks = np.stack([math.sqrt(w) * _unitary(rng, 4) for w in (0.7, 0.3)])
        out.append(("kraus", ks, (p[4], p[2]), ()))  # two-qubit channel
        for k in (3, 4, 5):
            out.append(("gate", _unitary(rng, 1 << k), tuple(int(x) for x in rng.permutation(n)[:k]), ()))
        ks = np.stack([math.sqrt(w) * _unitary(rng, 8) for w in (0.8, 0.15, 0.05)])
        out.append(("kraus", ks, tuple(int(x) for x in rng.permutation(n)[:3]), ()))  # three-qubit channel
    return out


def _experiment_kraus(rng, n, paths, p=0.8, eps=0.2):
    """The multiverse noise step as one Kraus set: the ideal path and, per noise path, a Pauli on one qubit and
    (two qubits and up) Paulis on two."""
    def place(hits):
        m = np.eye(1, dtype=C128)
        for x in range(n):
            m = np.kron(m, ONE[hits[x]] if x in hits else np.eye(2))
        return m

    out = [math.sqrt(p) * np.eye(1 << n, dtype=C128)]
    for _ in range(paths):
        out.append(math.sqrt(eps * 0.95 / paths) * place({int(rng.integers(n)): "XYZ"[int(rng.integers(3))]}))
        a, b = (int(x) for x in rng.choice(n, size=2, replace=False))
        out.append(math.sqrt(eps * 0.05 / paths) * place({a: "XYZ"[int(rng.integers(3))], b: "XYZ"[int(rng.integers(3))]}))
    return np.stack(out)


def _algorithm_gate(step, n):
    """The GHZ chain's gate of a step: H on the first qubit, then CNOTs from it."""
    return (ONE["H"], (0,)) if step % n == 0 else (CNOT, (0, step % n))


def _inputs(case, seed):
    """Everything a case's path is given, drawn from the seed alone (host side)."""
    rng = np.random.default_rng([seed, 1101])
    kind = case["kind"]
    if kind == "circuit":
        return {"ops": _circuit_ops(rng, case["n"], case["gates"], case["mix"], case["noise"]), "u": float(rng.uniform()),
                "qubit": int(rng.integers(case["n"])), "keep": sorted(int(x) for x in rng.choice(case["n"], 2, False))}
    if kind == "wide":
        return {"ops": _wide_ops(rng, case["n"], case["rounds"])}
    if kind == "experiment":
        return {"kraus": [_experiment_kraus(rng, case["n"], case["paths"]) for _ in range(case["steps"])]}
    if kind == "multiverse":
        n, v = case["n"], case["vectors"]
        w = rng.uniform(0.5, 1.5, v)
        return {"weights": w / w.sum(), "omegas": np.stack([np.eye(2), ONE["X"], ONE["Y"], ONE["Z"]]).astype(C128),
                "gates": [(_su2(rng), (int(rng.integers(n)),)) if s % 2 else
                          (CNOT, tuple(int(x) for x in rng.choice(n, size=2, replace=False))) for s in range(case["steps"])],
                "noise": [(int(rng.integers(n)), rng.choice(4, size=v, p=[0.8, 0.08, 0.06, 0.06]).astype(np.int32))
                          for _ in range(case["steps"])],
                "spread": [(_su2(rng), x) for x in range(n)]}
    if kind == "observables":
        n = case["n"]
        return {"pair": tuple(int(x) for x in rng.choice(n, 2, False)), "u": float(rng.uniform()), "qubit": int(rng.integers(n)),
                "keep": [sorted(int(x) for x in rng.choice(n, k, False)) for k in (1, 2, case["keep"])]}
    sizes = np.random.default_rng([ord(c) for c in kind] + [v for v in case.values() if isinstance(v, int)])
    if kind == "batch":  # register sizes and depths belong to the case, what the circuits hold to the seed
        ns = [min(8, case["nmax"])] + [int(x) for x in sizes.integers(case["nmin"], case["nmax"] + 1, case["circuits"] - 1)]
        return {"circuits": [Circuit(n, _circuit_ops(rng, n, int(sizes.integers(case["dmin"], case["dmax"] + 1)), "mixed",
                                                     "adpd", float(rng.uniform(0.001, 0.05)))) for n in ns]}
    w = 2.0 ** -np.arange(case["nmax"] - case["nmin"] + 1)
    ns = case["nmin"] + sizes.choice(len(w), size=case["requests"], p=w / w.sum())
    return {"circuits": [Circuit(int(n), _circuit_ops(rng, int(n), int(sizes.integers(case["dmin"], case["dmax"] + 1)),
                                                      "mixed", ("adpd", "dep", "none")[int(sizes.integers(3))])) for n in ns]}


def _chunks(ops, chunk):
    """The op list cut after every `chunk` gates (0: one piece)."""
    if not chunk:
        return [ops]
    out, cur, seen = [], [], 0
    for op in ops:
        if op.kind == "gate":
            if seen and seen % chunk == 0:
                out.append(cur)
                cur = []
            seen += 1
        cur.append(op)
    return out + [cur]


def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    st = {"case": case, "x": x}
    if kind in ("circuit", "wide", "experiment", "observables"):
        n = case["n"]
        rho = torch.zeros(1 << n, 1 << n, dtype=torch.complex64, device="cuda")
        st["rho"], st["d"] = rho, q.Density.from_tensor(rho)
        if kind in ("wide", "observables") or case.get("init") == "matrix":
            st["rho0"] = _density_matrix(n, seed)
        if kind == "circuit":
            if case["fused"]:
                st["d"].set_mode(q.QCW_MODE_FUSED, 0)
            st["packed"] = [q.PackedOps(c) for c in _chunks(x["ops"], case["chunk"])]
    elif kind == "multiverse":
        n = case["n"]
        e = q.Ensemble(n, case["vectors"])
        rho = torch.zeros(1 << n, 1 << n, dtype=torch.complex64, device="cuda")
        st.update(e=e, rho=rho, d=q.Density.from_tensor(rho))
        for u, t in x["spread"]:  # vectors with weight everywhere, as after the first gates of an algorithm
            e.apply_gate1(u, t)
    elif kind == "batch":
        st["b"] = q.Batch(x["circuits"])
    else:
        st["s"] = q.Server(1 << 28)
        st["packed"] = [q.PackedOps(c.ops) for c in x["circuits"]]
    return st


# ----------------------------------------------------------------------------- the path


def _f(v):
    v = np.asarray(v)
    return v.astype(np.complex64 if v.dtype.kind == "c" else np.float32)


def run(st):
    return globals()["_run_" + st["case"]["kind"]](st["case"], st["x"], st)


def _start(st):
    """The state every pass starts from: |0..0><0..0|, or the given matrix written into the caller's tensor."""
    if "rho0" in st:
        st["d"].device_state()
        st["rho"].copy_(st["rho0"])
    else:
        st["d"].reset()


def _run_circuit(case, x, st):
    d = st["d"]
    _start(st)
    tickets = []
    for p in st["packed"]:
        d.apply_packed(p)
        tickets.append(d.checkpoint())
    out = {"checkpoints": []}
    for t in tickets:
        tr, pu, p1 = d.checkpoint_read(t)
        out["checkpoints"].append([_f(tr.real), _f(pu), _f(p1)])
    out["reduced"] = _f(d.partial_trace(x["keep"]))
    if case["n"] <= 12:  # small registers end in the ancilla read-out
        m, p = d.measure(x["qubit"], -1, x["u"])
        out["outcome"], out["p"] = int(m), _f(p)
    d.device_state()
    out["rho"] = st["rho"]
    return out


def _run_wide(case, x, st):
    d = st["d"]
    _start(st)
    for call, m, qs, ctrl in x["ops"]:
        if call == "gate1":
            d.apply_gate1(m, qs[0], ctrl)
        elif call == "gate2":
            d.apply_gate2(m, qs[0], qs[1], ctrl)
        elif call == "gate":
            d.apply_gate(m, qs)
        else:
            d.apply_kraus(m, qs)
    d.device_state()
    return {"rho": st["rho"]}


def _run_experiment(case, x, st):
    d, n = st["d"], case["n"]
    _start(st)
    steps = []
    for s, ks in enumerate(x["kraus"]):
        d.apply_kraus(ks, range(n))
        u, qs = _algorithm_gate(s, n)
        if len(qs) == 1:
            d.apply_gate1(u, qs[0])
        else:
            d.apply_gate2(u, qs[0], qs[1])
        steps.append(np.concatenate([[d.purity()], d.polarization().ravel(), d.eigenvalues(range(n))]))
    d.device_state()
    return {"steps": _f(np.stack(steps)), "rho": st["rho"]}


def _run_multiverse(case, x, st):
    e, d = st["e"], st["d"]
    every = max(1, case["steps"] // case["densities"])
    purity = []
    for s, ((t, choice), (u, qs)) in enumerate(zip(x["noise"], x["gates"])):
        e.apply_noise1(x["omegas"], t, choice)
        if len(qs) == 1:
            e.apply_gate1(u, qs[0])
        else:
            e.apply_gate2(u, qs[0], qs[1])
        if (s + 1) % every == 0 or s + 1 == case["steps"]:
            e.density(x["weights"], d)
            purity.append(d.purity())
    d.device_state()
    return {"purity": _f(purity), "rho": st["rho"]}


def _run_observables(case, x, st):
    d = st["d"]
    _start(st)
    out = {"trace": _f(d.trace().real), "purity": _f(d.purity()), "p1": _f(d.probabilities()), "pol": _f(d.polarization()),
           "corr": _f(d.correlation(*x["pair"])), "reduced": [_f(d.partial_trace(k)) for k in x["keep"]],
           "entropy": _f(d.entropy(x["keep"][1])), "eig": _f(d.eigenvalues(x["keep"][2]))}
    m, p = d.measure(x["qubit"], -1, x["u"])
    out["outcome"], out["p"] = int(m), _f(p)
    d.device_state()
    out["rho"] = st["rho"]
    return out


def _run_batch(case, x, st):
    b = st["b"]
    b.run()
    p1, purity, trace = b.results()
    return {"p1": _f(np.concatenate(p1)), "purity": _f(purity), "trace": _f(trace), "state": _f(b.get_state(0))}


def _run_serve(case, x, st):
    s = st["s"]
    ids = [s.submit(c, p) for c, p in zip(x["circuits"], st["packed"])]
    s.drain()
    got = {r["id"]: r for r in s.poll()}
    return {"p1": _f(np.concatenate([got[i]["p1"] for i in ids])), "purity": _f([got[i]["purity"] for i in ids]),
            "trace": _f([got[i]["trace"] for i in ids])}


# ----------------------------------------------------------------------------- what it cannot do without


def _circuit_flops(n, ops):
    """One real 4 x 4 map per element for the one-qubit maps between two-qubit gates (two per such gate, one per qubit
    at the start); the two-qubit gates are permutations."""
    return 8.0 * 4.0 ** n * (2 * sum(1 for o in ops if o.k == 2) + n)


def work(case):
    kind = case["kind"]
    if kind == "circuit":
        n, el = case["n"], 4.0 ** case["n"]
        ops = _inputs(case, 0)["ops"]
        if case["fused"]:
            return {"bytes": 8 * el * (2 if case["init"] == "matrix" else 1), "flops": _circuit_flops(n, ops)}
        return {"bytes": 16 * el * len(ops), "flops": sum(2.0 * 4 ** o.k * el for o in ops if o.k == 1)}
    if kind == "wide":  # each call reads and writes the matrix once; a controlled gate touches what its controls select
        el, r = 4.0 ** case["n"], case["rounds"]
        return {"bytes": 16 * el * r * (0.44 + 0.75 + 0.75 + 6), "flops": el * r * 8 * sum(2 * 2 ** k for k in (2, 3, 4, 5, 3, 3, 3))}
    if kind == "experiment":
        el = 4.0 ** case["n"]
        return {"bytes": case["steps"] * (16 * el + 16 * el * (2 * case["paths"] + 1)),
                "flops": case["steps"] * (2 * case["paths"] + 1) * 16 * el * 2 ** case["n"]}
    if kind == "multiverse":
        n, v = case["n"], case["vectors"]
        nd = len([s for s in range(case["steps"]) if (s + 1) % max(1, case["steps"] // case["densities"]) == 0 or s + 1 == case["steps"]])
        return {"bytes": 32.0 * v * 2 ** n * case["steps"] + nd * (8 * 4.0 ** n + 8.0 * v * 2 ** n), "flops": nd * 4.0 * v * 4.0 ** n}
    if kind == "observables":
        return {"bytes": (16 + 4 + 8) * 4.0 ** case["n"], "flops": 4.0 * 4.0 ** case["n"]}
    x = _inputs(case, 0)["circuits"]
    return {"bytes": sum(8 * 4.0 ** c.n for c in x), "flops": sum(_circuit_flops(c.n, c.ops) for c in x)}


# ----------------------------------------------------------------------------- the same in 64 bits

DEV = "cuda" if torch.cuda.is_available() else "cpu"


def _zero(n):
    r = torch.zeros(1 << n, 1 << n, dtype=torch.complex128, device=DEV)
    r[0, 0] = 1
    return r


def _one_map(rho, n, t, s):
    """rho <- the one-qubit map s[(r, c), (r', c')] on qubit t."""
    v = rho.view(1 << t, 2, 1 << (n - 1 - t), 1 << t, 2, 1 << (n - 1 - t))
    old = [[v[:, r, :, :, c].clone() for c in (0, 1)] for r in (0, 1)]
    for r in (0, 1):
        for c in (0, 1):
            acc = v[:, r, :, :, c]
            acc.zero_()
            for a in (0, 1):
                for b in (0, 1):
                    z = complex(s[2 * r + c, 2 * a + b])
                    if z:
                        acc.add_(old[a][b], alpha=z)


def _kraus_map(ks):
    return sum(np.kron(k, k.conj()) for k in ks)


def _side(rho, n, m, qs, cols):
    """m on the row labels (or conj(m) on the column labels) of the qubits qs."""
    k = len(qs)
    t = rho.view([2] * (2 * n))
    ax = [x + (n if cols else 0) for x in qs]
    order = ax + [i for i in range(2 * n) if i not in ax]
    m = torch.as_tensor(np.asarray(m).conj() if cols else np.asarray(m), dtype=torch.complex128, device=rho.device)
    y = (m @ t.permute(order).reshape(1 << k, -1)).view([2] * (2 * n))
    inv = [order.index(i) for i in range(2 * n)]
    return y.permute(inv).reshape(1 << n, 1 << n).contiguous()


def _dense(rho, n, ks, qs):
    out = None
    for k in ks:
        y = _side(_side(rho, n, k, qs, False), n, k, qs, True)
        out = y if out is None else out.add_(y)
    return out


def _swap_elements(rho, n, gate, qs):
    """CNOT or CZ on both sides, in place."""
    for cols in (False, True):
        t = rho.view([2] * (2 * n))
        o = n if cols else 0
        on = [slice(None)] * (2 * n)
        on[qs[0] + o] = 1
        sub = t[tuple(on)]
        ax = qs[1] + o - (1 if qs[1] > qs[0] else 0)
        if gate is CNOT or np.array_equal(gate, CNOT):
            a, b = sub.select(ax, 0), sub.select(ax, 1)
            keep = a.clone()
            a.copy_(b)
            b.copy_(keep)
        else:
            sub.select(ax, 1).neg_()


def _exact_circuit(rho, n, ops):
    """The circuit in place; the one-qubit operations between two-qubit gates are multiplied together first."""
    pend = {}

    def flush(t):
        if t in pend:
            _one_map(rho, n, t, pend.pop(t))

    for o in ops:
        if o.k == 1:
            pend[o.qubits[0]] = _kraus_map(o.mats) @ pend.get(o.qubits[0], np.eye(4))
        else:
            for t in o.qubits:
                flush(t)
            _swap_elements(rho, n, o.mats[0], o.qubits)
    for t in list(pend):
        flush(t)


def _p1(rho, n):
    p = rho.diagonal().real.reshape([2] * n)
    return np.array([float(p.select(t, 1).sum()) for t in range(n)])


def _tr(rho):
    return float(rho.diagonal().real.sum())


def _purity(rho):
    return float(torch.view_as_real(rho).square().sum())


def _reduced(rho, n, keep):
    ax = [x for x in range(n) if x not in keep]
    t = rho.view([2] * (2 * n)).permute([*keep, *[n + x for x in keep], *ax, *[n + x for x in ax]])
    k, m = 1 << len(keep), 1 << len(ax)
    return torch.einsum("abii->ab", t.reshape(k, k, m, m)).cpu().numpy()


def _measured(rho, n, t, u):
    p1 = _p1(rho, n)[t]
    p0 = _tr(rho) - p1
    m = 0 if u < p0 else 1
    p = p1 if m else p0
    v = rho.view(1 << t, 2, 1 << (n - 1 - t), 1 << t, 2, 1 << (n - 1 - t))
    keep = v[:, m, :, :, m] / p
    rho.zero_()
    v[:, m, :, :, m] = keep
    return m, p


def _paulis(rho, n, strings):
    out = []
    for s in strings:  # Tr[P rho], one non-zero of P per row
        r = torch.arange(1 << n, device=rho.device)
        flip, val = 0, torch.ones(1 << n, dtype=torch.complex128, device=rho.device)
        for t, p in s:
            bit = (r >> (n - 1 - t)) & 1
            if p in "XY":
                flip |= 1 << (n - 1 - t)
            if p == "Y":
                val = val * torch.where(bit == 0, -1j, 1j)
            if p == "Z":
                val = val * (1 - 2 * bit)
        out.append(float((val * rho[r ^ flip, r]).sum().real))
    return np.array(out)


def _polarization(rho, n):
    return _paulis(rho, n, [[(t, p)] for t in range(n) for p in "XYZ"]).reshape(n, 3)


def exact(case, seed):
    x, kind = _inputs(case, seed), case["kind"]
    if kind == "circuit":
        n = case["n"]
        rho = _density_matrix(n, seed).to(torch.complex128) if case["init"] == "matrix" else _zero(n)
        out = {"checkpoints": []}
        for ops in _chunks(x["ops"], case["chunk"]):
            _exact_circuit(rho, n, ops)
            out["checkpoints"].append([np.float64(_tr(rho)), np.float64(_purity(rho)), _p1(rho, n)])
        out["reduced"] = _reduced(rho, n, x["keep"])
        if n <= 12:
            m, p = _measured(rho, n, x["qubit"], x["u"])
            out["outcome"], out["p"] = m, np.float64(p)
        out["rho"] = rho
        return out
    if kind == "wide":
        n = case["n"]
        rho = _density_matrix(n, seed).to(torch.complex128)
        for call, m, qs, ctrl in x["ops"]:
            if call == "kraus":
                rho = _dense(rho, n, m, qs)
                continue
            d = m.shape[0]
            full = np.eye(d << len(ctrl), dtype=C128)
            full[-d:, -d:] = m
            rho = _dense(rho, n, [full], [*ctrl, *qs])
        return {"rho": rho}
    if kind == "experiment":
        n = case["n"]
        rho, steps = _zero(n), []
        for s, ks in enumerate(x["kraus"]):
            rho = _dense(rho, n, ks, list(range(n)))
            u, qs = _algorithm_gate(s, n)
            rho = _dense(rho, n, [u], list(qs))
            ev = np.linalg.eigvalsh(rho.cpu().numpy())
            steps.append(np.concatenate([[_purity(rho)], _polarization(rho, n).ravel(), ev]))
        return {"steps": np.stack(steps), "rho": rho}
    if kind == "multiverse":
        n, v = case["n"], case["vectors"]
        psi = torch.zeros(v, 1 << n, dtype=torch.complex128, device=DEV)
        psi[:, 0] = 1

        def gate(u, qs, vec=None):
            nonlocal psi
            u = torch.as_tensor(u, dtype=torch.complex128, device=DEV)
            order = [0] + [1 + t for t in qs] + [1 + i for i in range(n) if i not in qs]
            t = psi.view([v] + [2] * n).permute(order).reshape(v, 1 << len(qs), -1)
            t = torch.matmul(u if vec is None else u[vec], t).view([v] + [2] * n)
            psi = t.permute([order.index(i) for i in range(n + 1)]).reshape(v, 1 << n).contiguous()

        for u, t in x["spread"]:
            gate(u, (t,))
        w = torch.as_tensor(x["weights"], dtype=torch.complex128, device=DEV)
        every, purity, rho = max(1, case["steps"] // case["densities"]), [], None
        for s, ((t, choice), (u, qs)) in enumerate(zip(x["noise"], x["gates"])):
            gate(x["omegas"], (t,), torch.as_tensor(choice, device=DEV).long())
            gate(u, qs)
            if (s + 1) % every == 0 or s + 1 == case["steps"]:
                rho = (psi * w[:, None]).T @ psi.conj()
                purity.append(_purity(rho))
        return {"purity": np.array(purity), "rho": rho}
    if kind == "observables":
        n = case["n"]
        rho = _density_matrix(n, seed).to(torch.complex128)
        red = [_reduced(rho, n, k) for k in x["keep"]]
        ev = [np.linalg.eigvalsh(0.5 * (r + r.conj().T)) for r in red]
        pos = ev[1][ev[1] > 1e-15]
        a, b = x["pair"]
        out = {"trace": np.float64(_tr(rho)), "purity": np.float64(_purity(rho)), "p1": _p1(rho, n), "pol": _polarization(rho, n),
               "corr": _paulis(rho, n, [[(a, i), (b, j)] for i in "XYZ" for j in "XYZ"]).reshape(3, 3), "reduced": red,
               "entropy": np.float64(-(pos * np.log2(pos)).sum()), "eig": ev[2]}
        m, p = _measured(rho, n, x["qubit"], x["u"])
        out["outcome"], out["p"], out["rho"] = m, np.float64(p), rho
        return out
    p1, purity, trace, state = [], [], [], None
    for c in x["circuits"]:
        rho = _zero(c.n)
        _exact_circuit(rho, c.n, c.ops)
        p1.append(_p1(rho, c.n))
        purity.append(_purity(rho))
        trace.append(_tr(rho))
        state = rho.cpu().numpy() if state is None else state
    out = {"p1": np.concatenate(p1), "purity": np.array(purity), "trace": np.array(trace)}
    return {**out, "state": state} if kind == "batch" else out
