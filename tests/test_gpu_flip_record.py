"""Rounds too large for the record of levels keep their flips instead: the
joint that reads them gives what the joint that runs the chains again gives
(which the oracle tests pin), element by element -- rows of one to four
words, ragged last words, both generation forms, rounds just past the
record's limit, weights under which most chains keep nothing and under which
all keep nearly everything, and both joint orders.
"""
import numpy as np
import pytest

import paper_0812_2964_gb300 as mc
from paper_0812_2964_gb300.workloads import random_weights

pytestmark = pytest.mark.gpu

LIMIT = 2 ** 33      # samples of the largest round whose levels are recorded


def _run(L, p, S, W, order, replay):
    g = mc.Job(L, p, 17 * L, 1)
    if replay:
        g.set_round_record(0)
    g.set_join_order(order)
    g.weights = W
    g.set_segment_samples(max(1 << 14, 2 * L * L))      # (the same checkpoints either way)
    out = []
    for _ in range(2):
        g.run_sweeps(S)
        kept = g.join()
        info = g.info()
        out.append((kept, g.hist, g.k, g.offsets, g.energies, info["carry_energy"], info["last_rejected"]))
        g.update_weights()
    held = g.info()["device_bytes"]
    g.close()
    return out, held


@pytest.mark.parametrize("L,p,S,scale,order", [(8, 9001, 15_000, 6.0, 0), (12, 1500, 40_000, 2.0, 0), (20, 9000, 2_400, 3.0, 1),
                                               (32, 8200, 1_030, 4.0, 0), (36, 2001, 3_350, 0.2, 0),
                                               (64, 1000, 2_150, 4.0, 0), (76, 700, 2_150, 0.2, 1),
                                               (100, 301, 2_900, 3.0, 0), (128, 160, 3_300, 0.3, 0)])
def test_flip_record_gives_the_replayed_joint(L, p, S, scale, order):
    samples = p * S * L * L
    assert LIMIT < samples < 1.2 * LIMIT
    W = random_weights(L, seed=L, scale=scale)
    a, held = _run(L, p, S, W, order, replay=False)
    b, held_replay = _run(L, p, S, W, order, replay=True)
    for x, y in zip(a, b):
        for u, v in zip(x, y):
            assert np.array_equal(u, v)
    # a bit a sample, every chain's words padded to whole lines
    words = -(-S * L * ((L + 31) // 32) // 32) * 32
    assert held - held_replay == 4 * p * words
    assert held == mc.mc_job_device_bytes(L, p, S)
