"""GPU parity of the one-pass kernel for operations on three to five qubits (gates and channels, one
or several operators per launch, operators spread over blocks or summed over launches) against the
oracle."""

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
