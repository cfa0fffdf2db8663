"""Every form of generation writes the same flip record: rows of one to four
words one chain a lane (in shared and in global memory, in groups of four
lanes) and one a warp a word at a time, each against the joint that runs the
chains again (bit for bit); and generation on a caller's buffers where the
lattices are swept in place."""
import numpy as np
import pytest

import paper_0812_2964_gb300 as mc
from paper_0812_2964_gb300.workloads import random_weights

pytestmark = pytest.mark.gpu

LIMIT = 2 ** 33      # samples of the largest round whose levels are recorded


def _round(L, p, S, W, shape, replay):
    g = mc.Job(L, p, 13 * L, 1)
    if replay:
        g.set_round_record(0)
    if shape is not None:
        g.set_launch_shape(*shape)
    g.weights = W
    g.run_sweeps(S)
    kept = g.join()
    out = (kept, g.hist, g.k, g.offsets, g.energies, g.info()["carry_energy"])
    held = g.info()["device_bytes"]
    g.close()
    return out, held


@pytest.mark.parametrize("L,p,S,shape", [
    (32, 4100, 2_050, (1, 1, 4)), (20, 9000, 2_400, (1, 1, 4)),                    # one a warp, one word
    (100, 1300, 670, (1, 1, 4)), (128, 1300, 410, (1, 1, 4)),                      # four words, a word at a time
    (24, 9000, 1_670, (1, 32, 4)), (36, 4100, 1_620, (1, 32, 4)),                  # lanes, lattices in shared memory
    (64, 4100, 515, (1, 32, 4)), (96, 4100, 230, (1, 16, 4)), (128, 4100, 130, (1, 12, 4)),
    (48, 4100, 920, (1, 8, 4)), (64, 4100, 515, (1, 4, 4)), (96, 4100, 230, (1, 8, 4)), (128, 4100, 130, (1, 8, 4)),
    (96, 6200, 155, (2, 32, 4)), (100, 4100, 215, (2, 16, 4)), (128, 4100, 130, (2, 32, 4)),   # in global memory
    (100, 4100, 215, (2, 8, 4)), (128, 4100, 130, (2, 4, 4)),
    (64, 8200, 260, None)])                                                        # past the default's line
def test_forms_keep_the_same_flips(L, p, S, shape):
    assert LIMIT < p * S * L * L < 1.2 * LIMIT
    W = random_weights(L, seed=L + 2, scale=2.0)
    a, held = _round(L, p, S, W, shape, replay=False)
    b, held_replay = _round(L, p, S, W, None if shape is None else (1, 2, 1), replay=True)
    for u, v in zip(a, b):
        assert np.array_equal(u, v)
    words = -(-S * L * ((L + 31) // 32) // 32) * 32
    assert held >= held_replay + 4 * p * words                 # (the flips were there)


@pytest.mark.parametrize("L,p", [(96, 6200), (100, 9800), (128, 4900)])
def test_noalloc_with_lattices_swept_in_place(L, p):
    torch = pytest.importorskip("torch")
    N, seed = L * L, 77 + L
    W = random_weights(L, seed=L, scale=3.0)
    job = mc.Job(L, p, seed, 1)
    assert job.info()["placement"] == 2
    job.set_launch_shape(1, 1, 4)                              # (the other side: one chain a warp)
    job.weights = W
    dev = torch.device("cuda")
    d_spins = torch.from_numpy(job.spin_words.reshape(-1).view(np.int32).copy()).to(dev)
    d_levels = torch.from_numpy(((job.energies + 2 * N) // 4).astype(np.int32)).to(dev)
    d_W = torch.from_numpy(W.astype(np.float64)).to(dev)
    d_hist = torch.zeros(N + 1, dtype=torch.int64, device=dev)
    torch.cuda.synchronize()
    job.run_sweeps(1)
    job.join_naive()
    mc.mc_generate_noalloc(L, p, seed, 0, 1, d_spins.data_ptr(), d_levels.data_ptr(), d_W.data_ptr(),
                           d_hist.data_ptr(), None)
    torch.cuda.synchronize()
    assert np.array_equal(d_spins.cpu().numpy().view(np.uint32), job.spin_words.reshape(-1))
    assert np.array_equal(d_levels.cpu().numpy(), (job.energies + 2 * N) // 4)
    assert np.array_equal(d_hist.cpu().numpy(), job.hist)
    job.close()


def test_graph_batch_of_kept_and_replayed_rounds_on_a_users_stream():
    torch = pytest.importorskip("torch")
    groups = [(16, 70, 21), (32, 50, 22), (64, 33, 23), (20, 40, 24)]
    st = torch.cuda.Stream()

    def jobs():
        js = [mc.Job(L, p, s, 1) for L, p, s in groups]
        js[1].set_round_record(0)          # replayed beside kept ones
        js[3].set_round_record(0)
        return js

    js = jobs()
    js[0].set_stream(st.cuda_stream)
    js[2].set_stream(st.cuda_stream)
    mc.mc_batch_run(js, 3, 4, 2)
    for j, k in zip(js, jobs()):
        for _ in range(3):
            k.run_sweeps(4)
            k.join()
            k.update_weights()
        assert np.array_equal(j.weights, k.weights)
        assert np.array_equal(j.spin_words, k.spin_words)
        j.close()
        k.close()


def test_a_few_rejections_do_not_send_a_flip_round_to_the_heights():
    # young weights: once between a sixteenth and a quarter of the chains are rejected, the next joint still
    # searches first (the scan then settles what the passes left, not every chain), with the replayed results
    L, p, S = 64, 2048, 1_100
    assert LIMIT < p * S * L * L < 1.2 * LIMIT
    rounds = []
    for replay in (False, True):
        g = mc.Job(L, p, 3, 1)
        if replay:
            g.set_round_record(0)
        out, before = [], 0
        for _ in range(6):
            g.run_sweeps(S)
            kept = g.join()
            info = g.info()
            out.append((kept, g.hist, g.k, info["carry_energy"]))
            if not replay and p // 16 < before <= p // 4:
                assert info["last_scanned"] < p
                out.append("smooth enough")
            before = info["last_rejected"]
            g.update_weights()
        g.close()
        rounds.append(out)
    assert "smooth enough" in [x for x in rounds[0] if isinstance(x, str)]
    for a, b in zip([x for x in rounds[0] if not isinstance(x, str)], rounds[1]):
        for u, v in zip(a, b):
            assert np.array_equal(u, v)
