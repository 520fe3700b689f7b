"""CPU tests of the Pauli-basis planner: its passes, replayed on the Pauli coefficients of a
random state the way the kernel walks them (tiles, rounds, swizzled positions), must give the
coefficients of the oracle's state after the original operations."""

import ctypes
import itertools
import os
import subprocess

import numpy as np
import pytest

import oracle
import workloads as wl
from tests._helpers import haar_unitary, random_rho

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1101_1785_gb300", "csrc")
PAULI = [np.eye(2), np.diag([1, -1]), np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]])]  # label 2 x + z


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("pauli") / "libpauli_shim.so")
    src = [os.path.join(CSRC, f) for f in ("planner.cpp", "tile.cpp", "pauli_plan.cpp")]
    src.append(os.path.join(os.path.dirname(os.path.abspath(__file__)), "cpp", "pauli_shim.cpp"))
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    "-I", "/usr/local/cuda/include", "-o", out, *src], check=True)
    return ctypes.CDLL(out)


def coefficients(rho):
    """Tr[P rho] for every string, index = base-4 digits with qubit n - 1 lowest (flattened)."""
    n = rho.shape[0].bit_length() - 1
    t = rho.reshape([2] * (2 * n))
    for q in range(n):  # row axis of the first qubit left is 0, its column axis n - q; labels go last
        t = np.moveaxis(t, [0, n - q], [0, 1])
        t = np.stack([np.einsum("cr,rc...->...", p, t) for p in PAULI], axis=-1)
    return np.ascontiguousarray(t.real.reshape(-1))


def test_coefficient_helper():
    rho = random_rho(np.random.default_rng(0), 3)
    v = coefficients(rho)
    for i, lab in enumerate(itertools.product(range(4), repeat=3)):
        p = np.kron(np.kron(PAULI[lab[0]], PAULI[lab[1]]), PAULI[lab[2]])
        assert abs(np.trace(p @ rho) - v[i]) < 1e-12


def _packed(ops):
    kind, k, qs, mats, off = [], [], [], [], []
    pos = 0
    for op in ops:
        if op.kind == "gate":
            m = op.mats[0]
        else:
            m = sum(np.kron(a, a.conj()) for a in op.mats)
        kind.append(0 if op.kind == "gate" else 1)
        k.append(len(op.qubits))
        qs += (list(op.qubits) + [0])[:2]
        off.append(pos)
        mats.append(np.ascontiguousarray(m, dtype=np.complex128).ravel())
        pos += mats[-1].size
    I = lambda a: np.asarray(a, dtype=np.int32)
    kind, k, qs, off = I(kind), I(k), I(qs), np.asarray(off, dtype=np.int64)
    mats = np.concatenate(mats)
    return kind, k, qs, mats, off


def _replay(shim, n, ops, v, kmax, beam, zero=False):
    kind, k, qs, mats, off = _packed(ops)
    nr, bad = ctypes.c_int(), ctypes.c_int()
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    npass = shim.pauli_replay(n, kmax, int(beam), int(zero), len(ops), p(kind), p(k), p(qs), p(mats), p(off), p(v),
                              ctypes.byref(nr), ctypes.byref(bad))
    assert npass > 0 and bad.value == 0
    return npass


def _two_qubit_ops(rng, n, count):
    ops = []
    for i in range(count):
        a, b = (int(x) for x in rng.permutation(n)[:2])
        kind = i % 5
        if kind == 0:
            ops.append(wl.Op("gate", (a, b), haar_unitary(rng, 4)[None]))
        elif kind == 1:
            ops.append(wl.Op("kraus", (a, b), np.stack([np.sqrt(w) * haar_unitary(rng, 4) for w in (0.6, 0.3)])))
        elif kind == 2:
            ops.append(wl.Op("gate", (a, b), wl.gate_matrix("CNOT")[None]))
        elif kind == 3:
            ops.append(wl.Op("gate", (a, b), wl.gate_matrix("CZ")[None]))
        else:  # target before control in the list
            x = wl.gate_matrix("CNOT")
            s = wl.gate_matrix("SWAP")
            ops.append(wl.Op("gate", (a, b), (s @ x @ s)[None]))
        q = int(rng.integers(n))
        ops.append(wl.Op("kraus", (q,), np.stack([np.sqrt(0.5) * haar_unitary(rng, 2), 0.4 * haar_unitary(rng, 2)])))
        ops.append(wl.Op("gate", (q,), haar_unitary(rng, 2)[None]))
    return ops


@pytest.mark.parametrize("n,kmax,beam", [(3, 0, 0), (4, 2, 0), (5, 0, 0), (6, 5, 0), (7, 0, 0), (8, 0, 0), (8, 3, 1), (9, 0, 1)])
@pytest.mark.parametrize("what", ["mixed", "haar70", "two"])
def test_plan_replays_the_circuit(shim, n, kmax, beam, what):
    rng = np.random.default_rng(100 * n + kmax)
    if what == "two":
        ops = _two_qubit_ops(rng, n, 25)
    else:
        ops = wl.random_circuit(n, 60, 17 * n + kmax, what, "adpd" if what == "mixed" else "dep").ops
    rho = random_rho(rng, n)
    v = coefficients(rho)
    want = rho.copy()
    for op in ops:
        oracle.apply_op(want, op)
    _replay(shim, n, ops, v, kmax, beam)
    # FP32 coefficients of the composed maps: 2^-24 relative each, at most a few per operation kept
    scale = np.linalg.norm(coefficients(want))
    assert np.linalg.norm(v - coefficients(want)) <= len(ops) * 2.0 ** -24 * scale


@pytest.mark.parametrize("n", [3, 5, 8])
@pytest.mark.parametrize("what", ["mixed", "two", "ones"])
def test_plan_from_the_zero_state(shim, n, what):
    """One-qubit operations before the first two-qubit one go into the product state the plan starts
    from (all of them, when there is no two-qubit operation)."""
    rng = np.random.default_rng(n)
    ops = _two_qubit_ops(rng, n, 12) if what == "two" else wl.random_circuit(n, 50, 5 + n, "mixed", "adpd").ops
    if what == "ones":
        ops = [op for op in ops if op.k == 1]
    want = wl.zero_state(n)
    for op in ops:
        oracle.apply_op(want, op)
    v = np.zeros(4 ** n)
    _replay(shim, n, ops, v, 0, False, True)
    assert np.linalg.norm(v - coefficients(want)) <= (len(ops) + n) * 2.0 ** -24 * np.linalg.norm(coefficients(want))


@pytest.mark.parametrize("n", [1, 2, 3, 5, 6])
@pytest.mark.parametrize("what", ["mixed", "haar70", "two", "ones"])
def test_plain_list_passes(shim, n, what):
    """The plain path's passes over a list (runs on two qubits, dense two-qubit maps, maps left over)."""
    rng = np.random.default_rng(7 * n)
    if n == 1 or what == "ones":
        ops = [wl.Op("gate", (int(rng.integers(n)),), haar_unitary(rng, 2)[None]) for _ in range(9)]
    elif what == "two":
        ops = _two_qubit_ops(rng, n, 30)
    else:
        ops = wl.random_circuit(n, 80, 9 + n, what, "adpd" if what == "mixed" else "dep").ops
    rho = random_rho(rng, n)
    v = coefficients(rho)
    want = rho.copy()
    for op in ops:
        oracle.apply_op(want, op)
    kind, k, qs, mats, off = _packed(ops)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    passes = shim.pairs_replay(n, len(ops), p(kind), p(k), p(qs), p(mats), p(off), p(v))
    assert 0 < passes < len(ops)
    assert np.linalg.norm(v - coefficients(want)) <= len(ops) * 2.0 ** -24 * np.linalg.norm(coefficients(want))


def _list_differs(shim, n, ops):
    kind, k, qs, mats, off = _packed(ops)
    raw = np.concatenate([np.ascontiguousarray(op.mats, dtype=np.complex128).ravel() for op in ops])
    sizes = [len(op.mats) * 4 ** len(op.qubits) for op in ops]
    raw_off = np.asarray(np.cumsum([0] + sizes[:-1]), dtype=np.int64)
    nk = np.asarray([len(op.mats) for op in ops], dtype=np.int32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    return shim.list_plan_differs(n, len(ops), p(kind), p(k), p(qs), p(mats), p(off), p(raw), p(nk), p(raw_off))


def _depolarising(q, f):
    """The channel that scales the polarisation of qubit q by f."""
    w = [(1 + 3 * f) / 4] + [(1 - f) / 4] * 3
    return wl.Op("kraus", (q,), np.stack([np.sqrt(a) * p for a, p in zip(w, PAULI)]).astype(complex))


@pytest.mark.parametrize("count", [1, 60, 140, 185, 195, 210, 300])
def test_vanishing_maps_leave_later_ones_alone(shim, count):
    """A long run of depolarising channels (a map whose linear part falls to and below the smallest FP32
    numbers) on a qubit that is used again afterwards: the maps that follow keep their own scale."""
    n, f = 3, 0.6
    c01 = wl.Op("gate", (0, 1), wl.gate_matrix("CNOT")[None])
    ops = [c01] + [_depolarising(0, f)] * count + [c01, wl.Op("gate", (0,), wl.gate_matrix("H")[None])]
    want = wl.zero_state(n)
    for op in ops:
        oracle.apply_op(want, op)
    want = coefficients(want)
    tol = 16 * 2.0 ** -24  # a few roundings of coefficients at most 1
    v = np.zeros(4 ** n)
    _replay(shim, n, ops, v, 0, False, True)
    assert np.abs(v - want).max() <= tol
    v = coefficients(wl.zero_state(n))
    _replay(shim, n, ops, v, 0, False)
    assert np.abs(v - want).max() <= tol
    v = coefficients(wl.zero_state(n))
    kind, k, qs, mats, off = _packed(ops)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    assert shim.pairs_replay(n, len(ops), p(kind), p(k), p(qs), p(mats), p(off), p(v)) > 0
    assert np.abs(v - want).max() <= tol
    assert _list_differs(shim, n, ops) == 0


@pytest.mark.parametrize("scale", [1.0, 1e-4, 1e-8, 1e-12, 1e6])
def test_small_operators_are_kept(shim, scale):
    """One-qubit operators far from unit norm (an unnormalised branch of a channel): what counts as the
    residue of an exact zero is measured against the map's own largest entry."""
    rng = np.random.default_rng(3)
    n = 3
    ops = [wl.Op("gate", (0,), scale * haar_unitary(rng, 2)[None]), wl.Op("gate", (0, 2), wl.gate_matrix("CNOT")[None]),
           wl.Op("kraus", (2,), scale * np.stack([np.sqrt(w) * haar_unitary(rng, 2) for w in (0.7, 0.2)])),
           wl.Op("gate", (0, 1), wl.gate_matrix("CZ")[None]), wl.Op("gate", (1,), haar_unitary(rng, 2)[None])]
    want = random_rho(rng, n)
    v0 = coefficients(want)
    for op in ops:
        oracle.apply_op(want, op)
    want = coefficients(want)
    tol = 16 * 2.0 ** -24 * np.abs(want).max()
    v = v0.copy()
    _replay(shim, n, ops, v, 0, False)
    assert np.abs(v - want).max() <= tol
    v = v0.copy()
    kind, k, qs, mats, off = _packed(ops)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    assert shim.pairs_replay(n, len(ops), p(kind), p(k), p(qs), p(mats), p(off), p(v)) > 0
    assert np.abs(v - want).max() <= tol
    assert _list_differs(shim, n, ops) == 0


@pytest.mark.parametrize("n,kmax", [(8, 0), (9, 0), (10, 0), (8, 3), (10, 5)])
def test_no_pass_without_operations(shim, n, kmax):
    """A pass cut at its program's limits leaves operations to later ones; sets of the beam search that
    find nothing left to do are not run."""
    for seed in range(12):
        rng = np.random.default_rng(100 * n + seed)
        ops = []
        for i in range(60):  # dense maps on few qubits fill a pass's program, the others wait for them
            few = rng.permutation(min(n, 4))[:2] if i % 3 else rng.permutation(n)[:2]
            ops.append(wl.Op("gate", tuple(int(x) for x in few), haar_unitary(rng, 4)[None]))
        kind, k, qs, mats, off = _packed(ops)
        p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        npass = ctypes.c_int()
        assert shim.pauli_empty_passes(n, kmax, 1, len(ops), p(kind), p(k), p(qs), p(mats), p(off), ctypes.byref(npass)) == 0
        assert npass.value > 1
    rho = random_rho(rng, n)
    v = coefficients(rho)
    for op in ops:
        oracle.apply_op(rho, op)
    _replay(shim, n, ops, v, kmax, True)
    want = coefficients(rho)
    assert np.linalg.norm(v - want) <= 2 * len(ops) * 2.0 ** -24 * np.linalg.norm(want)
