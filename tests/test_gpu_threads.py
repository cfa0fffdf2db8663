"""Host threads with a job each: kernels that jobs of every size share are
launched from both at once, and each thread's results are those it has alone
(whole rounds of recorded levels, rounds of a few attempts, averages)."""
import threading

import numpy as np
import pytest

import paper_0812_2964_gb300 as mc
from paper_0812_2964_gb300.workloads import random_weights

pytestmark = pytest.mark.gpu

BETAS = np.linspace(0.1, 1.0, 305)      # (past the count up to which small lattices use another kernel)


def _work(L, p, seed, turns):
    """One digest a turn; every turn starts from the same state, so all agree."""
    out = []
    for _ in range(turns):
        g = mc.Job(L, p, seed, 1)
        g.weights = random_weights(L, seed, 2.0)
        g.visited = np.ones(L * L + 1, np.uint8)
        got = [g.thermo(BETAS)]
        for _ in range(4):
            g.run_sweeps(2)
            got += [g.join(), g.hist, g.k]
        got.append(g.thermo(BETAS))
        for _ in range(3):
            g.run_attempts(60)
            got += [g.join(), g.k]
        got += [g.thermo(BETAS), g.energies]
        g.close()
        out.append(got)
    return out


def test_threads_with_jobs_of_different_sizes():
    mc.build()
    specs = [(16, 300, 3), (64, 40, 4), (128, 20, 5), (20, 100, 6)]
    alone = [_work(*s, 1)[0] for s in specs]
    got, errors = {}, []

    def run(i):
        try:
            got[i] = _work(*specs[i], 60)
        except Exception as e:          # (a thread's exception reaches the test through the list)
            errors.append((specs[i], repr(e)))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(specs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for i, want in enumerate(alone):
        for turn in got[i]:
            for a, b in zip(turn, want):
                assert np.array_equal(a, b)
