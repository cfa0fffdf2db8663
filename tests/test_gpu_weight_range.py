"""Weights far outside a grown job's range: the joints of kept rounds give what
the replaying joint gives when weights mask levels with huge values, when a
level no chain visits carries one, and when whole ranges are lifted; the
averages of weights that are all huge are the oracle's."""
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


def _rows(up):
    """bool [p][L][L], L <= 32 -> the job's words."""
    p, L, _ = up.shape
    return (up.astype(np.uint32) << np.arange(L, dtype=np.uint32)).sum(2, dtype=np.uint32).reshape(-1)


def _same(a, b):
    for x, y in zip(a, b):
        for u, v in zip(x, y):
            assert np.array_equal(u, v)


@pytest.mark.parametrize("mask", [-1e30, -1e300, -8.9e307])
def test_masked_levels(mask):
    # two masks, the deeper one on the antiferromagnetic side: chains that start below the first and above the
    # second stay there (every move among equal weights is taken: one wall sweeps through the lattice, at most
    # 9 of 64 levels from the end), and the round's input is a masked level while chain 0 is not
    L, p = 8, 96
    N = L * L
    W = random_weights(L, 5, 0.5)
    W[:12], W[53:] = mask, 2 * mask
    stripes = np.add.outer(np.arange(L), np.arange(L)) % 2 == 0
    up = np.ones((p, L, L), bool)
    up[p // 2:-1] = stripes
    mixed = np.random.default_rng(1).random((L, L)) < 0.5

    def run(replay):
        g = mc.Job(L, p, 9, 0)
        if replay:
            g.set_round_record(0)
        g.weights = W
        g.spin_words = _rows(up)
        out = []
        for r in range(4):
            g.run_sweeps(3)
            kept = g.join()
            out.append((kept, g.hist, g.k, g.energies, g.info()["carry_energy"], g.info()["last_rejected"]))
            if r == 0:                                   # half the chains rejected: the next joint is by heights
                assert g.info()["last_rejected"] == p // 2 - 1
                words = g.spin_words.reshape(p, L).copy()
                words[0] = _rows(mixed[None])
                g.spin_words = words.reshape(-1)
                g.set_join_order(1)
        g.close()
        return out

    _same(run(False), run(True))


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("extra", [7.2e5, -7.2e5, 1e8, -1e12, 3e38, -1e300, np.inf, -np.inf])
def test_a_level_nobody_visits(extra, order):
    # level 1 does not exist on the lattice: whatever its weight, the joint is that of the other levels
    L, p, S = 12, 1500, 4
    W = random_weights(L, 6, 5.0)

    def run(replay, w1):
        g = mc.Job(L, p, 10, 1)
        if replay:
            g.set_round_record(0)
        w = W.copy()
        w[1] = w1
        g.weights = w
        g.set_join_order(order)
        out = []
        for _ in range(4):
            g.run_sweeps(S)
            out.append((g.join(), g.hist, g.k, g.offsets, g.energies, g.info()["carry_energy"]))
        g.close()
        return out

    want = run(True, extra)
    _same(run(False, extra), want)
    _same(run(True, 0.0), want)


@pytest.mark.parametrize("attempts", [False, True])
@pytest.mark.parametrize("lift", [1e6, 1e9, -1e9])
def test_levels_lifted_out_of_the_filters_range(lift, attempts):
    # half the levels far above (below) the level that the heights are measured against, with the usual
    # differences among themselves: answers come from the exact test alone
    L, p = 12, 700
    W = random_weights(L, 7, 4.0)
    W[L * L // 2:] += lift

    def run(fast):
        g = mc.Job(L, p, 11, 1)
        if not fast:
            g.set_round_record(0)
            g.set_partial_record(0)
        g.weights = W
        out = []
        for _ in range(4):
            g.run_attempts(70) if attempts else g.run_sweeps(2)
            out.append((g.join(), g.hist, g.k, g.offsets, g.energies, g.info()["carry_energy"]))
        g.close()
        return out

    _same(run(True), run(False))


def test_rough_joints_of_many_chains_are_settled_by_the_heights():
    # every input of a joint after a rough one is the heights' answer: none is left to the pass that
    # searches whole chains (the scan counts the chains it settled)
    L, p = 8, 1 << 17
    g = mc.Job(L, p, 12, 1)
    g.weights = random_weights(L, 8, 8.0)
    settled = []
    for r in range(9):
        g.run_sweeps(1)
        g.join()
        info = g.info()
        assert info["last_rejected"] > p // 16
        if r:
            settled.append(info["last_scanned"])
    g.close()
    assert settled == [p] * 8


def test_an_undecided_chain_does_not_end_the_scan():
    # the weight of a level nobody visits widens the error bound (to 0.01): of the same joints some then have an
    # undecided chain, which is searched and the scan goes on behind it -- no pass searches whole chains
    L, p = 8, 1 << 17
    out, passes = [], []
    for w1 in (0.0, 28_000.0):
        g = mc.Job(L, p, 12, 1)
        w = random_weights(L, 8, 8.0)
        w[1] = w1
        g.weights = w
        rounds = []
        for _ in range(9):
            g.run_sweeps(1)
            rounds.append((g.join(), g.hist, g.k, g.energies, g.info()["carry_energy"]))
            passes.append(g.info()["last_passes"])
        out.append(rounds)
        g.close()
    _same(*out)
    assert max(passes) <= 5


@pytest.mark.parametrize("L,n", [(8, 5), (16, 305), (36, 7)])
@pytest.mark.parametrize("base", [1e39, -1e39, 3.3e38, 1e300])
def test_thermo_of_huge_weights(L, n, base):
    N = L * L
    W = np.full(N + 1, base)
    W[1::3] = base * (1 + 2.0 ** -50)
    vis = np.ones(N + 1, np.uint8)
    vis[::5] = 0
    betas = np.linspace(0.05, 1.0, n)
    g = mc.Job(L, 2, 1, 1)
    g.weights = W
    g.visited = vis
    a, b = g.thermo(betas), oracle.thermo(L, W, vis, betas)
    g.close()
    assert np.isfinite(b).all()
    assert np.allclose(a[:, 0], b[:, 0], rtol=1e-10, atol=1e-10 * N)
    assert np.allclose(a[:, 1], b[:, 1], rtol=1e-9, atol=1e-9 * N)
    assert np.allclose(a[:, 2], b[:, 2], rtol=1e-10)
    assert np.allclose(a[:, 3], b[:, 3], rtol=0, atol=1e-10 * max(N, abs(base)))


@pytest.mark.parametrize("L,n", [(12, 9), (36, 9), (64, 300)])
def test_thermo_of_infinite_weights(L, n):
    # a whole stretch of visited levels without any share: it adds nothing
    N = L * L
    W = random_weights(L, 4, 2.0)
    W[N // 2:3 * N // 4] = np.inf
    vis = np.ones(N + 1, np.uint8)
    betas = np.linspace(0.05, 1.0, n)
    g = mc.Job(L, 2, 1, 1)
    g.weights = W
    g.visited = vis
    a, b = g.thermo(betas), oracle.thermo(L, W, vis, betas)
    g.close()
    assert np.isfinite(b).all()
    assert np.allclose(a[:, 0], b[:, 0], rtol=1e-10, atol=1e-10 * N)
    assert np.allclose(a[:, 1], b[:, 1], rtol=1e-9, atol=1e-9 * N)
    assert np.allclose(a[:, 2], b[:, 2], rtol=1e-10)
    assert np.allclose(a[:, 3], b[:, 3], rtol=0, atol=1e-10 * N)
