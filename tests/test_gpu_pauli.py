"""GPU parity of Pauli storage (the default fused path from 3 qubits up) against the oracle: the
pass kernel at every tile size it takes, the changes of basis in both directions, the readouts on
the Pauli coefficients, and the storage changes between fused, plain and direct use."""

import numpy as np
import pytest

import oracle
import workloads as wl
from tests._helpers import haar_unitary, random_rho

pytestmark = pytest.mark.gpu

ATOL = 1e-5
READ_TOL = 1e-6


@pytest.fixture(scope="module")
def q():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1101_1785_gb300 as q

    return q


def _apply(d, ops):
    for op in ops:
        d.apply_op(op)


def _dense_ops(rng, n, count):
    """Every operation kind of the pass kernel: CNOT both ways, CZ, dense gates and channels,
    one-qubit maps that lose trace."""
    ops = []
    x = wl.gate_matrix("CNOT")
    s = wl.gate_matrix("SWAP")
    for i in range(count):
        a, b = (int(v) for v in rng.permutation(n)[:2])
        m = (x, wl.gate_matrix("CZ"), s @ x @ s, haar_unitary(rng, 4), s)[i % 5]
        ops.append(wl.Op("gate", (a, b), m[None]))
        if i % 4 == 0:
            ops.append(wl.Op("kraus", (b, a), np.stack([np.sqrt(w) * haar_unitary(rng, 4) for w in (0.7, 0.28)])))
        t = int(rng.integers(n))
        ops.append(wl.Op("gate", (t,), haar_unitary(rng, 2)[None]))
        if i % 3 == 0:
            ops.append(wl.Op("kraus", (t,), np.stack([np.sqrt(0.6) * haar_unitary(rng, 2), 0.6 * haar_unitary(rng, 2)])))
    return ops


@pytest.mark.parametrize("n,k", [(3, 0), (4, 0), (5, 0), (6, 0), (7, 0), (8, 0), (8, 3), (9, 0), (10, 5)])
@pytest.mark.parametrize("what", ["mixed", "haar70", "dense"])
def test_state_and_readouts(q, n, k, what):
    rng = np.random.default_rng(40 * n + k)
    ops = _dense_ops(rng, n, 20) if what == "dense" else wl.random_circuit(n, 90, 300 + n, what, "adpd").ops
    for start in ("zero", "matrix"):
        d = q.Density(n)
        d.set_mode(q.QCW_MODE_FUSED, k)
        want = wl.zero_state(n) if start == "zero" else random_rho(rng, n)
        if start == "matrix":
            d.set_state(want)
        else:
            d.reset()
        _apply(d, ops)
        for op in ops:
            oracle.apply_op(want, op)
        assert abs(d.trace() - oracle.trace(want)) <= READ_TOL
        assert abs(d.purity() - oracle.purity(want)) <= READ_TOL
        np.testing.assert_allclose(d.probabilities(), oracle.probabilities(want), atol=READ_TOL, rtol=0)
        for keep in ([0], [0, n - 1], list(range(min(n, 6))), list(range(n))):
            if len(keep) <= 8:
                np.testing.assert_allclose(d.partial_trace(keep), oracle.partial_trace(want, keep), atol=READ_TOL, rtol=0)
        got = d.get_state()
        assert np.abs(got - want).max() <= ATOL
        if start == "zero":  # changed back from Pauli storage: both triangles from the same numbers
            assert np.abs(got - got.conj().T).max() == 0.0
        # again from the matrix the state was changed back to
        _apply(d, ops)
        for op in ops:
            oracle.apply_op(want, op)
        pol = d.polarization()
        assert np.abs(pol - oracle.polarization(want)).max() <= READ_TOL
        m_ref, p_ref = oracle.measure(want, n - 1, 1)
        m, p = d.measure(n - 1, 1)
        assert m == m_ref and abs(p - p_ref) <= READ_TOL
        assert abs(d.purity() - oracle.purity(want)) <= ATOL
        m_ref, p_ref = oracle.measure(want, 0, 0)
        m, p = d.measure(0, 0)
        assert m == m_ref and abs(p - p_ref) <= ATOL
        assert np.abs(d.get_state() - want).max() <= ATOL
        d.close()


@pytest.mark.parametrize("n", [3, 5, 7, 8, 11, 13])
def test_change_of_basis_round_trip(q, n):
    """rho -> Pauli coefficients -> rho through circuits that undo themselves, against the state."""
    rng = np.random.default_rng(n)
    psi = rng.standard_normal((1 << n, 2)) + 1j * rng.standard_normal((1 << n, 2))
    rho = psi @ psi.conj().T
    rho /= np.trace(rho).real
    d = q.Density(n)
    d.set_mode(q.QCW_MODE_FUSED, 0)
    d.set_state(rho)
    x = wl.gate_matrix("CNOT")
    pairs = [tuple(int(v) for v in rng.permutation(n)[:2]) for _ in range(30)]
    for a, b in pairs + pairs[::-1]:
        d.apply_gate2(x, a, b)
    got = d.get_state()
    # the passes only rename coefficients: the error is that of the two transforms, at most
    # 2 n additions of 2^-24 relative per element of a vector of the state's norm
    assert np.linalg.norm(got - rho) <= 4 * n * 2.0 ** -24 * np.linalg.norm(rho)
    d.close()


def test_storage_changes_between_modes(q):
    """Fused work, a wide gate (plain), plain mode, device access, reset and fused work again."""
    n = 8
    rng = np.random.default_rng(5)
    c = wl.random_circuit(n, 60, 11, "mixed", "adpd")
    d = q.Density(n)
    d.set_mode(q.QCW_MODE_FUSED, 0)
    assert np.abs(d.get_state() - wl.zero_state(n)).max() == 0.0
    d.reset()
    assert d.trace() == 1.0 and d.purity() == 1.0 and (d.probabilities() == 0).all()
    want = wl.zero_state(n)
    u3 = haar_unitary(rng, 8)
    for part in range(3):
        _apply(d, c.ops)
        for op in c.ops:
            oracle.apply_op(want, op)
        d.apply_gate(u3, [5, 0, 3])
        oracle.apply_unitary(want, u3, [5, 0, 3])
        if part == 1:
            d.set_mode(q.QCW_MODE_PLAIN, 0)
        if part == 2:
            d.device_state()
            d.set_mode(q.QCW_MODE_FUSED, 0)
    _apply(d, c.ops)
    for op in c.ops:
        oracle.apply_op(want, op)
    assert np.abs(d.get_state() - want).max() <= ATOL
    d.set_fused_kernel(3)
    _apply(d, c.ops)
    d.set_fused_kernel(0)
    _apply(d, c.ops)
    for op in c.ops + c.ops:
        oracle.apply_op(want, op)
    assert abs(d.purity() - oracle.purity(want)) <= ATOL
    assert np.abs(d.get_state() - want).max() <= ATOL
    d.close()


@pytest.mark.parametrize("n", [12, 14])
def test_many_tiles_per_block_are_reproducible(q, n):
    """Dozens of tiles per thread block: every run from |0..0> gives the same bits, and the purity
    summed by the last pass agrees with the one taken from the matrix."""
    c = wl.random_circuit(n, 120, 1400 + n, "mixed", "adpd")
    p = q.PackedOps(c.ops)
    d = q.Density(n)
    d.set_mode(q.QCW_MODE_FUSED, 0)
    seen = []
    for _ in range(8):
        d.reset()
        d.apply_packed(p)
        seen.append((d.purity(), d.probabilities()))
    for pu, pr in seen[2:]:  # the second run plans again (beam search)
        assert pu == seen[1][0]
        np.testing.assert_array_equal(pr, seen[1][1])
    assert abs(seen[0][0] - seen[1][0]) <= READ_TOL
    d.device_state()
    assert abs(d.purity() - seen[1][0]) <= READ_TOL
    d.close()


def test_wait_that_runs_out_is_reported(q):
    n = 9
    c = wl.random_circuit(n, 60, 404, "mixed", "adpd")
    d = q.Density(n)
    d.set_mode(q.QCW_MODE_FUSED, 0)
    d.reset()
    d.set_fused_wait_limit(2000, 0)  # the first CTA skips the load of its first tile
    _apply(d, c.ops)
    with pytest.raises(q.QcwError) as e:
        d.trace()
    assert e.value.status == q.QCW_ETIMEOUT
    d.set_fused_wait_limit(0, -1)
    d.reset()
    _apply(d, c.ops)
    assert np.abs(d.get_state() - oracle.run_circuit(c)).max() <= ATOL
    d.close()


@pytest.mark.parametrize("n", [3, 4, 7])
@pytest.mark.parametrize("gates", [3, 300])
def test_small_registers_stay_on_rho(q, n, gates):
    """A state of up to seven qubits given as a matrix is evolved as one, however long the circuit: a
    population far below the others keeps its relative precision where nothing acts on its qubit."""
    rng = np.random.default_rng(n)
    p = 1e-9
    psi = np.zeros(2 ** n, complex)
    psi[0], psi[2 ** (n - 1)] = np.sqrt(1 - p), np.sqrt(p)
    d = q.Density(n)
    d.set_mode(q.QCW_MODE_FUSED)
    d.set_state(np.outer(psi, psi))
    for i in range(gates):
        d.apply_gate(haar_unitary(rng, 2), (1 + i % (n - 1),))
        if n > 2:
            a, b = (int(x) for x in 1 + rng.permutation(n - 1)[:2])
            d.apply_gate2(wl.gate_matrix("CNOT"), a, b)
    # FP32: every operation rounds an element a few times, in either direction
    assert abs(d.probabilities()[0] - p) <= 2 * gates * 8 * 2.0 ** -24 * p
    assert d.measure(0, 1)[0] == 1


@pytest.mark.parametrize("n,touched,gates", [(8, 7, 11), (8, 8, 40), (9, 2, 1), (9, 2, 60), (10, 7, 70), (11, 11, 20), (9, 4, 5)])
@pytest.mark.parametrize("k", [0, 3])
def test_storage_of_a_given_matrix(q, n, touched, gates, k):
    """Either side of the rule that says when a matrix is changed to Pauli storage."""
    rng = np.random.default_rng(n + touched)
    want = random_rho(rng, n, 3)
    d = q.Density(n)
    d.set_mode(q.QCW_MODE_FUSED, k)
    d.set_state(want)
    where = rng.permutation(n)[:touched]
    ops = []
    for i in range(gates):
        a, b = (int(x) for x in rng.permutation(where)[:2])
        ops.append(wl.Op("gate", (a, b), (haar_unitary(rng, 4) if i % 3 == 0 else wl.gate_matrix("CNOT"))[None]))
        ops.append(wl.Op("kraus", (a,), np.stack([np.sqrt(0.7) * haar_unitary(rng, 2), np.sqrt(0.3) * haar_unitary(rng, 2)])))
    for _ in range(2):
        _apply(d, ops)
        for op in ops:
            oracle.apply_op(want, op)
        np.testing.assert_allclose(d.probabilities(), oracle.probabilities(want), atol=READ_TOL, rtol=0)
        assert np.abs(d.get_state() - want).max() <= ATOL


def test_storage_is_tried_again_for_the_next_state(q):
    """Without room for the coefficients the passes run on rho; once there is room, the next state takes them."""
    import torch

    n = 15  # rho 8 GiB, the coefficients 4 GiB
    d = q.Density(n)
    d.set_mode(q.QCW_MODE_FUSED)
    held, left = [], 2 << 30
    while torch.cuda.mem_get_info()[0] > left + (64 << 20):
        free = torch.cuda.mem_get_info()[0] - left
        held.append(torch.empty(min(free, 8 << 30) // (2 << 20) * (2 << 20), dtype=torch.uint8, device="cuda"))
    d.reset()
    d.apply_gate1(wl.gate_matrix("H"), 0)
    d.apply_gate2(wl.gate_matrix("CNOT"), 0, n - 1)
    assert abs(d.correlation(0, n - 1)[2, 2] - 1) <= READ_TOL
    held.clear()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    d.reset()
    d.apply_gate1(wl.gate_matrix("H"), 0)
    d.apply_gate2(wl.gate_matrix("CNOT"), 0, n - 1)
    assert abs(d.correlation(0, n - 1)[2, 2] - 1) <= READ_TOL
    assert before - torch.cuda.mem_get_info()[0] >= 4 << 30
    d.close()


@pytest.mark.parametrize("how", ["fused", "list", "batch"])
@pytest.mark.parametrize("theta", [1e-2, 1e-3, 3e-4, 1e-4, 0.0])
def test_small_probabilities(q, how, theta):
    """Probabilities near 0: a weak rotation, and (theta = 0) operations that undo one another.  Absolute
    error of a few FP32 roundings of numbers at most 1; a forced outcome agrees with what was read."""
    rng = np.random.default_rng(4)
    n = 4
    op = lambda m, *qs: wl.Op("gate", qs, np.asarray(m, complex)[None])
    c, s = np.cos(theta / 2), np.sin(theta / 2)
    u, cx = haar_unitary(rng, 2), wl.gate_matrix("CNOT")
    ops = [op([[c, -s], [s, c]], 0), op(u, 1), op(cx, 1, 2), op(haar_unitary(rng, 2), 2), op(cx, 0, 3)]
    if theta == 0:
        ops = [op(u, 0), op(u, 1), op(cx, 0, 1), op(cx, 1, 3), op(cx, 1, 3), op(cx, 0, 1), op(u.conj().T, 1), op(u.conj().T, 0)]
    want = wl.zero_state(n)
    for o in ops:
        oracle.apply_op(want, o)
    want, tol = oracle.probabilities(want), 2.0 ** -22
    if how == "batch":
        b = q.Batch([wl.Circuit(n, ops)])
        b.run()
        assert np.abs(b.results()[0][0] - want).max() <= tol
        return
    d = q.Density(n)
    if how == "fused":
        d.set_mode(q.QCW_MODE_FUSED)
        d.reset()
    d.apply_packed(q.PackedOps(ops))
    got = d.probabilities()
    assert np.abs(got - want).max() <= tol
    if got[0] >= 1e-12:
        assert d.measure(0, 1) == (1, got[0])
    else:
        with pytest.raises(q.QcwError) as err:
            d.measure(0, 1)
        assert err.value.status == q.QCW_EZEROPROB
    d.close()
