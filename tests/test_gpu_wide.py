"""GPU parity of the one-pass kernel for operations on three to five qubits (gates and channels, one
or several operators per launch, operators spread over blocks or summed over launches) and of the
warp-per-output partial trace, against the oracle; operation lists on the plain path against the same
operations one by one."""

import numpy as np
import pytest

import oracle
import workloads as wl
from tests._helpers import haar_unitary, random_rho

pytestmark = pytest.mark.gpu

ATOL = 1e-5


@pytest.fixture(scope="module")
def q():
    import __graft_entry__

    __graft_entry__.build()
    import paper_1101_1785_gb300 as q

    return q


# (n, k, operators): n = k (one tile); operators spread over blocks; one launch; several launches
# that collect the sum (a launch carries 48, 12 and 3 operators of 3, 4 and 5 qubits)
@pytest.mark.parametrize("n,k,nk", [(3, 3, 1), (3, 3, 50), (4, 3, 2), (9, 3, 3), (9, 3, 49), (4, 4, 13), (7, 4, 1), (9, 4, 13),
                                    (5, 5, 17), (6, 5, 1), (8, 5, 4), (10, 5, 4), (10, 5, 1)])
def test_wide_operations(q, n, k, nk):
    rng = np.random.default_rng(1000 * n + 100 * k + nk)
    rho = random_rho(rng, n)
    want = rho.copy()
    d = q.Density(n)
    d.set_state(rho)
    for _ in range(2):
        qs = [int(x) for x in rng.permutation(n)[:k]]
        if nk == 1:
            u = haar_unitary(rng, 1 << k)
            d.apply_gate(u, qs)
            oracle.apply_unitary(want, u, qs)
        else:
            w = rng.uniform(0.5, 1.5, nk)
            ks = np.stack([np.sqrt(x) * haar_unitary(rng, 1 << k) for x in w / w.sum()])
            d.apply_kraus(ks, qs)
            oracle.apply_kraus(want, ks, qs)
    assert np.abs(d.get_state() - want).max() <= ATOL
    assert abs(d.trace() - 1) <= 1e-6
    d.close()


@pytest.mark.parametrize("n,ntr", [(5, 5), (7, 5), (8, 6), (9, 7), (10, 8)])
@pytest.mark.parametrize("half", [False, True])
def test_partial_trace_shapes(q, n, ntr, half):
    """One output per thread, warp and block, on the full matrix and on its lower triangle."""
    rng = np.random.default_rng(10 * n + ntr)
    c = wl.random_circuit(n, 40, 70 + n, "mixed", "adpd")
    want = oracle.run_circuit(c)
    d = q.Density(n)
    if half and n >= 6:
        d.set_mode(q.QCW_MODE_FUSED, 4)
        d.set_fused_kernel(3)
    for op in c.ops:
        d.apply_op(op)
    for _ in range(3):
        keep = sorted(int(x) for x in rng.permutation(n)[: n - ntr])
        np.testing.assert_allclose(d.partial_trace(keep), oracle.partial_trace(want, keep), atol=1e-6, rtol=0)
    d.close()


@pytest.mark.parametrize("n,nvec", [(1, 3), (3, 2048), (5, 16), (5, 2049), (6, 4096), (7, 700), (8, 515), (9, 600)])
def test_density_shared_out_over_the_vectors(q, n, nvec):
    """Registers with few tiles: every block sums a share of the vectors.  A second noise step and
    density right behind the first (no host wait in between) must not disturb it."""
    rng = np.random.default_rng(100 * n + nvec)
    psi = rng.standard_normal((nvec, 1 << n)) + 1j * rng.standard_normal((nvec, 1 << n))
    psi /= np.linalg.norm(psi, axis=1)[:, None]
    psi = psi.astype(np.complex64).astype(np.complex128)
    w = rng.uniform(0.1, 1.0, nvec)
    w /= w.sum()
    om = np.stack([wl.gate_matrix("I"), wl.gate_matrix("X"), wl.gate_matrix("Z")])
    e = q.Ensemble(n, nvec)
    e.set(psi)
    ds = [q.Density(n), q.Density(n)]
    want = []
    for d in ds:
        t = int(rng.integers(n))
        pick = rng.integers(0, 3, nvec).astype(np.int32)
        e.apply_noise1(om, t, pick)
        v = psi.reshape(nvec, 1 << t, 2, -1)
        psi = np.einsum("vij,vajb->vaib", om[pick], v).reshape(nvec, -1)
        e.density(w, d)
        want.append((psi * w[:, None]).T @ psi.conj())
    for d, x in zip(ds, want):
        # FP32 products and sums of at most a few hundred terms of weight w |psi|^2 per block
        assert np.abs(d.get_state() - x).max() <= 32 * 2.0 ** -24 * np.abs(x).max()
        assert abs(d.trace() - 1) <= 1e-6
        d.close()
    e.close()


@pytest.mark.parametrize("n", [1, 2, 4, 6, 7, 8])
@pytest.mark.parametrize("what", ["mixed", "haar70", "all"])
def test_plain_lists(q, n, what):
    """A list in plain mode joins its neighbours (all of it in one launch up to six qubits, a pass per
    pair above); any matrix, not only a Hermitian one."""
    rng = np.random.default_rng(90 * n)
    if n == 1:
        ops = [wl.Op("kraus" if i % 3 == 0 else "gate", (0,), np.stack([0.8 * haar_unitary(rng, 2), 0.6 * haar_unitary(rng, 2)])
                     if i % 3 == 0 else haar_unitary(rng, 2)[None]) for i in range(12)]
    else:
        ops = wl.random_circuit(n, 150 if n < 7 else 60, 31 + n, "haar70" if what == "haar70" else "mixed", "adpd").ops
    if what == "all" and n > 1:  # dense gates and channels, permutations, wider operations, lost trace
        for i in range(0, 40, 4):
            a, b = (int(x) for x in rng.permutation(n)[:2])
            s = wl.gate_matrix("SWAP")
            ops.insert(3 * i, wl.Op("gate", (a, b), (s, haar_unitary(rng, 4), s @ wl.gate_matrix("CNOT") @ s)[i % 3][None]))
            ops.insert(3 * i, wl.Op("kraus", (b, a), np.stack([np.sqrt(0.6) * haar_unitary(rng, 4), 0.6 * haar_unitary(rng, 4)])))
            ops.insert(3 * i, wl.Op("kraus", (a,), np.stack([np.sqrt(0.6) * haar_unitary(rng, 2), 0.63 * haar_unitary(rng, 2)])))
            if n > 3:
                ops.insert(3 * i, wl.Op("gate", tuple(int(x) for x in rng.permutation(n)[:3]), haar_unitary(rng, 8)[None]))
    z = rng.standard_normal((1 << n, 1 << n)) + 1j * rng.standard_normal((1 << n, 1 << n))
    z /= np.linalg.norm(z)
    a, b = q.Density(n), q.Density(n)
    a.set_state(z), b.set_state(z)
    a.apply_packed(q.PackedOps(ops))
    for op in ops:
        b.apply_op(op)
    # a handful of FP32 roundings per operation on either side, of elements of norm at most 1
    assert np.abs(a.get_state() - b.get_state()).max() <= 8 * len(ops) * 2.0 ** -24
    assert a.stats()["launches"] < b.stats()["launches"]
    a.close(), b.close()


@pytest.mark.parametrize("n,k,nk,more", [(5, 5, 8, 33), (4, 3, 20, 64), (9, 3, 49, 60)])
def test_captured_channels_keep_their_scratch(q, n, k, nk, more):
    """A channel of many operators in a captured graph: the graph carries the operators, and a channel
    of more operators afterwards leaves the scratch it was captured with in place."""
    import torch

    rng = np.random.default_rng(10 * n + k)

    def channel(count):
        w = rng.uniform(0.5, 1.5, count)
        return np.stack([np.sqrt(x) * haar_unitary(rng, 1 << k) for x in w / w.sum()])

    qs = [int(x) for x in rng.permutation(n)[:k]]
    first, second = channel(nk), channel(more)
    start = random_rho(rng, n)
    s = torch.cuda.Stream()
    rho = torch.zeros(1 << n, 1 << n, dtype=torch.complex64, device="cuda")
    torch.cuda.synchronize()
    d = q.Density.from_tensor(rho, s)
    d.set_state(start)
    d.apply_kraus(first, qs)  # scratch and kernel attributes are there before the capture
    d.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        d.apply_kraus(first, qs)
    d.set_state(start)
    d.apply_kraus(second, qs)
    d.sync()
    held = torch.zeros(1 << 20, device="cuda")  # where memory given back would go
    with torch.cuda.stream(s):
        g.replay()
    want = start.copy()
    oracle.apply_kraus(want, second, qs)
    oracle.apply_kraus(want, first, qs)
    assert np.abs(d.get_state() - want).max() <= ATOL
    assert float(held.abs().max()) == 0.0
    d.close()
