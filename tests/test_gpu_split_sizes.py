"""Sizes on both sides of where the work is split another way: statistical
averages with and without a launch of their own for the normalisation (up to
L = 32 and 304 temperatures), and rounds of a few attempts joined by one block
(up to 4096 chains) or by several.  The averages to the tolerance of the other
thermo tests (the same sums in another order; C, a difference of squares of
order N, to 1e-9 N absolutely), the rounds bit for bit.
"""
import numpy as np
import pytest

import oracle
import paper_0812_2964_gb300 as mc
from paper_0812_2964_gb300.workloads import random_weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    mc.build()
    oracle.build()


@pytest.mark.parametrize("L,n", [(16, 304), (16, 305), (32, 1), (32, 305), (36, 10)])
def test_thermo(L, n):
    N = L * L
    W = random_weights(L, 3, 2.0)
    vis = np.ones(N + 1, dtype=np.uint8)
    vis[::7] = 0
    betas = np.linspace(0.01, 1.2, n)
    g = mc.Job(L, 2, 1, 1)
    g.weights = W
    g.visited = vis
    a, b = g.thermo(betas), oracle.thermo(L, W, vis, betas)
    assert np.allclose(a[:, 0], b[:, 0], rtol=1e-10, atol=1e-10 * N)
    assert np.allclose(a[:, 1], b[:, 1], rtol=1e-9, atol=1e-9 * N)
    assert np.allclose(a[:, 2], b[:, 2], rtol=1e-10)
    assert np.allclose(a[:, 3], b[:, 3], rtol=0, atol=1e-10 * N)


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("p", [4096, 4097, 9000])
def test_attempt_rounds(p, order):
    L, n = 8, 40
    W = random_weights(L, 8, 4.0)
    g, o = mc.Job(L, p, 3, 1), oracle.Job(L, p, 3, 1)
    g.weights = W
    o.weights = W
    g.set_join_order(order)
    o.set_join_order(order)
    for _ in range(3):
        g.run_attempts(n)
        o.run_attempts(n, 4)
        assert g.join() == o.join()
        assert np.array_equal(g.k, o.k)
        assert np.array_equal(g.hist, o.hist)
        assert g.info()["carry_energy"] == 4 * o.carry - 2 * L * L
