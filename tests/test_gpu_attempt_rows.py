"""Rounds of a few attempts move only the lattice rows they sweep and their
neighbours: rounds that begin and end inside a row, at its ends, around the
lattice's last row and just short of all rows, against the oracle, bit for
bit (rows of one and of two words)."""
import numpy as np
import pytest

import oracle
import paper_0812_2964_gb300 as mc
from paper_0812_2964_gb300.workloads import random_weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L", [4, 8, 36])
def test_rows_of_a_round(L):
    mc.build()
    oracle.build()
    N, p = L * L, 35
    W = random_weights(L, 4, 2.0)
    g, o = mc.Job(L, p, 6, 1), oracle.Job(L, p, 6, 1)
    g.weights = W
    o.weights = W
    at = 0
    for n in (1, L - 1, L, 1, 2 * L - 1, N - 2 * L - 1, L + 1, N - 2 * L, N - L - 1, 3, N - L, N - 1, 1, N + 3, L // 2,
              N - L + 1, 2 * N - 5):
        g.run_attempts(n)
        o.run_attempts(n, 4)
        at += n
        assert np.array_equal(g.spin_words, oracle.pack_spins(o.spins)), (n, at)
        assert np.array_equal(g.energies, 4 * o.levels - 2 * N)
        assert g.join() == o.join()
        assert np.array_equal(g.hist, o.hist)
    g.close()
