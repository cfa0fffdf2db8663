"""Memory that a call can do without does not make it fail: a record that
cannot be had leaves the round to the replaying joint, with the same
results.  (Allocation failures are injected on the host, before any CUDA call.)
"""
import time

import numpy as np
import pytest

import paper_0812_2964_gb300 as mc
from paper_0812_2964_gb300.workloads import random_weights

pytestmark = pytest.mark.gpu

MIB = 2 ** 20
BIG = (32, 8200, 1030)          # L, chains, sweeps: just too large for the record of levels
BIG_FLIPS = 4 * 8200 * 1030 * 32


@pytest.fixture(scope="module", autouse=True)
def _built():
    mc.build()
    yield
    mc.mc_inject_alloc_failure(-1)


def _alone(L, p, seed, iters, S, replay=False):
    g = mc.Job(L, p, seed, 1)
    if replay:
        g.set_round_record(0)
    for _ in range(iters):
        g.run_sweeps(S)
        g.join()
        g.update_weights()
    W = g.weights
    g.close()
    return W


# ------------------------------------------------------------------ one job
@pytest.mark.parametrize("after", [0, 1, 2, 3])
def test_flip_rounds_fall_back_to_replays(after):
    # 0..2: the checkpoints that rebuilding from flips wants, 3: the flips themselves
    L, p, S = BIG
    W = random_weights(L, 3, 1.0)
    out = []
    for replay in (False, True):
        g = mc.Job(L, p, 71, 1)
        g.weights = W
        if replay:
            g.set_round_record(0)
        else:
            mc.mc_inject_alloc_failure(after)
        g.run_sweeps(S)
        mc.mc_inject_alloc_failure(-1)
        kept = g.join()
        out.append((kept, g.hist, g.k, g.energies))
        if not replay:
            assert g.info()["device_bytes"] < mc.mc_job_device_bytes(L, p, S)    # (the flips are not there)
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


# ------------------------------------------------------------------ batches
BATCH = [(8, 40, 11), (16, 70, 12), (20, 50, 13)]      # L, chains, seed


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("after", [9, 10, 11])
def test_batch_records_come_after_what_every_job_needs(mode, after):
    # three checkpoint buffers a job first, then a record a job: a record that fails is done without
    live0 = mc.mc_live_allocations()
    js = [mc.Job(L, p, seed, 1) for L, p, seed in BATCH]
    mc.mc_inject_alloc_failure(after)
    mc.mc_batch_run(js, 2, 5, mode)
    mc.mc_inject_alloc_failure(-1)
    for j, (L, p, seed) in zip(js, BATCH):
        assert np.array_equal(j.weights, _alone(L, p, seed, 2, 5))
        j.close()
    assert mc.mc_live_allocations() == live0


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("after", [3, 5, 8])
def test_batch_reports_what_it_cannot_do_without(mode, after):
    js = [mc.Job(L, p, seed, 1) for L, p, seed in BATCH]
    mc.mc_inject_alloc_failure(after)
    with pytest.raises(mc.McError) as e:
        mc.mc_batch_run(js, 2, 5, mode)
    mc.mc_inject_alloc_failure(-1)
    assert e.value.code == mc.MC_ENOMEM
    mc.mc_batch_run(js, 2, 5, mode)                      # and the next call works
    for j, (L, p, seed) in zip(js, BATCH):
        assert np.array_equal(j.weights, _alone(L, p, seed, 2, 5))
        j.close()


# ------------------------------------------------------------------ serving
def test_server_runs_a_large_round_without_room_for_its_flips():
    L, p, S = BIG
    budget = mc.mc_job_device_bytes(L, p, S) - BIG_FLIPS
    with mc.Server(budget, max_slots=2) as srv:
        W, st = srv.wait(srv.submit(L, p, 81, 2, S))
        assert srv.info()["peak_bytes"] <= budget
    assert st["status"] == mc.MC_OK and st["device_bytes"] <= budget
    assert np.array_equal(W, _alone(L, p, 81, 2, S, replay=True))


def test_server_takes_flips_back_for_a_job_that_waits():
    L, p, S = BIG
    small = (64, 500, 82, 2, 3)
    budget = mc.mc_job_device_bytes(L, p, S) + MIB       # room for the large job whole, not for both
    assert mc.mc_job_device_bytes(64, 500, 3) > MIB
    with mc.Server(budget, max_slots=2) as srv:
        a = srv.submit(L, p, 83, 12, S)
        deadline = time.monotonic() + 60
        while srv.info()["bytes_in_use"] < mc.mc_job_device_bytes(L, p, S) and time.monotonic() < deadline:
            time.sleep(0.001)
        assert srv.info()["bytes_in_use"] == mc.mc_job_device_bytes(L, p, S)
        b = srv.submit(*small)
        Wb, stb = srv.wait(b)
        Wa, sta = srv.wait(a)
        assert srv.info()["peak_bytes"] <= budget and srv.info()["bytes_in_use"] == 0
    assert stb["t_admit"] < sta["t_done"]                # it did not wait for the large job's end
    assert np.array_equal(Wb, _alone(*small))
    assert np.array_equal(Wa, _alone(L, p, 83, 12, S, replay=True))


def test_server_keeps_flips_where_there_is_room():
    L, p, S = BIG
    need = mc.mc_job_device_bytes(L, p, S)
    with mc.Server(2 * need, max_slots=2) as srv:
        W, st = srv.wait(srv.submit(L, p, 84, 2, S))
    assert st["device_bytes"] == need
    assert np.array_equal(W, _alone(L, p, 84, 2, S))
