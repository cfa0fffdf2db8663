"""The joint's passes over recorded rounds that fill the chip: blocks of 4 to
12 warps (by how many of them an SM holds beside the level weights), lanes by
chain index whatever the joint's order, four samples a test.  Element by
element what the joint that runs the chains again gives (which the oracle
tests pin): weights under which most chains keep nothing and under which
nearly all keep something, both joint orders, segments with a ragged end.
"""
import numpy as np
import pytest

import paper_0812_2964_gb300 as mc
from paper_0812_2964_gb300.workloads import random_weights

pytestmark = pytest.mark.gpu


def _run(L, p, S, W, order, replay):
    g = mc.Job(L, p, 5 * L + 1, 1)
    if replay:
        g.set_round_record(0)
    g.set_join_order(order)
    g.weights = W
    out = []
    for _ in range(2):
        g.run_sweeps(S)
        kept = g.join()
        out.append((kept, g.hist, g.k, g.offsets, g.energies, g.info()["carry_energy"], g.info()["last_rejected"]))
        g.update_weights()
    g.close()
    return out


@pytest.mark.parametrize("L,p,S,scale,order", [(16, 4100, 170, 4.0, 1), (52, 1000, 77, 4.0, 1), (52, 1000, 77, 0.2, 0),
                                               (100, 1501, 13, 3.0, 1), (128, 1024, 11, 3.0, 0), (128, 1000, 11, 0.3, 1)])
def test_recorded_joint_gives_the_replayed_joint(L, p, S, scale, order):
    samples = p * S * L * L
    assert 2048 * 152 * 512 < samples < 2 ** 28      # segments of 2048 samples, more than the chip holds at once
    W = random_weights(L, seed=L + 1, scale=scale)
    for x, y in zip(_run(L, p, S, W, order, replay=False), _run(L, p, S, W, order, replay=True)):
        for u, v in zip(x, y):
            assert np.array_equal(u, v)
