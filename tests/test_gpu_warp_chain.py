"""Generation with one chain per warp (shape placement 1, one chain a warp)
against the oracle, element by element: row lengths from a fraction of a
warp to four words with a ragged last one, chain counts that leave the last
block part empty and that fill several blocks per SM, levels recorded and
not, and the weights that make the word's fixed point hardest to reach --
noise of the order of the thresholds themselves and a visited range that
ends in cliffs (any tolerance is zero: integers, and identical bits of W).
"""
import numpy as np
import pytest

from paper_0812_2964_gb300.workloads import random_weights
from test_gpu_parity import _run_parity

pytestmark = pytest.mark.gpu


def _cliffs(L):
    """A young weight: levels around the middle visited (W about -15), the rest untouched."""
    N = L * L
    W = np.zeros(N + 1)
    lo, hi = N // 2 - N // 8, N // 2 + N // 8
    W[lo:hi] = -15.0 + 0.2 * np.sin(np.arange(hi - lo))
    return W


@pytest.mark.parametrize("record", [True, False])
@pytest.mark.parametrize("L,p,S", [(4, 5, 9), (8, 33, 5), (12, 7, 4), (20, 9, 3), (28, 5, 2), (32, 6, 3), (36, 5, 2),
                                   (60, 3, 2), (64, 5, 2), (68, 3, 2), (96, 3, 2), (100, 3, 2), (124, 2, 2),
                                   (128, 3, 2)])
def test_row_lengths(L, p, S, record):
    for W in (random_weights(L, L, 4.0), _cliffs(L)):
        _run_parity(L, p, S, 2, 1, seed=100 + L, weights=W, shape=(1, 1, 1), record=record)


@pytest.mark.parametrize("p", [1, 152, 153, 607, 609, 1217, 2432])
def test_chain_counts(p):
    _run_parity(16, p, 1, 2, 1, seed=7, weights=random_weights(16, 2, 1.0), shape=(1, 1, 2))


def test_default_shape_is_one_chain_a_warp():
    _run_parity(48, 40, 2, 3, 1, seed=9)


@pytest.mark.parametrize("L", [36, 64, 68, 100, 128])
def test_many_chains_of_long_rows(L):
    """Past the chain count up to which rows are resolved 64 sites at a time."""
    _run_parity(L, 1300, 1, 2, 1, seed=11, weights=random_weights(L, 5, 3.0))
