"""The work that a user of paper_0812_2964_gb300 has it do, case by case, through its public
entry points (``Job``, ``mc_batch_run``, ``mc_thermo``, ``Server``, ``mc_generate_noalloc``).

A case is a dict of plain values with a ``kind``:

* ``iteration``  one weight iteration of one job: a round of S sweeps of every chain, the joint,
  the weight update; the user reads the histogram, the weights, the joint and the chains back.
  ``resume`` 1 starts from a weight already close to -ln g(E) (plus the noise of an estimate)
  with the chains spread over the energy range, as a job has them once its weight has grown;
  0 starts as ``mc_init`` does, from W = 0, so that repeated passes are a young job's iterations.
* ``attempts``   one round of a few attempts (less than a sweep) and its joint.
* ``noalloc``    one generation round on the caller's own device buffers.
* ``thermo``     the averages E, C, F, S on a curve of inverse temperatures.
* ``batch``      weight iterations of several jobs of different L in fused launches (CUDA graph).
* ``serving``    a burst of weight-estimation jobs through the continuous-batching server.
"""
from __future__ import annotations

import numpy as np
import torch

import paper_0812_2964_gb300 as mc
from paper_0812_2964_gb300.workloads import BATCH_GROUPS, serving_stream

# exact() runs every chain and every joint in plain numpy: only rounds this small
EXACT_ATTEMPTS = 8_000          # attempts per chain
EXACT_SAMPLES = 8_000_000       # attempts of all chains


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # Fig. 2's shape: rounds of M_node = 100 attempts at L = 20, joined each time -- a run
        # is 10^5 and more of these tiny rounds, so a call's latency is all there is
        {"name": "round_L20_p32_100", "kind": "attempts", "L": 20, "p": 32, "n": 100, "resume": 1},
        # part (ii): the averages on a temperature curve, asked again and again while a weight grows
        {"name": "thermo_L64_b200", "kind": "thermo", "L": 64, "betas": 200},
        # a small job as the serving stream has them: 20 sweeps a round
        {"name": "job_L16_p512_S20", "kind": "iteration", "L": 16, "p": 512, "S": 20, "start": 1,
         "resume": 1, "ordered": 0, "trace": 0},
        # generation for a caller that owns the buffers (and its own joint)
        {"name": "noalloc_L96_p1280_S20", "kind": "noalloc", "L": 96, "p": 1280, "S": 20},
        # an odd size: L that is no multiple of 32, a ragged chain count, energy-ordered joining
        {"name": "ordered_L52_p1000_S100", "kind": "iteration", "L": 52, "p": 1000, "S": 100, "start": 1,
         "resume": 1, "ordered": 1, "trace": 0},
        # the small configuration: 64 chains of 10^4 sweeps at L = 8
        {"name": "job_L8_p64_S10000", "kind": "iteration", "L": 8, "p": 64, "S": 10_000, "start": 0,
         "resume": 1, "ordered": 0, "trace": 0},
        # the paper's Table 1 run (Fig. 1): few long chains of a large lattice
        {"name": "job_L100_p32_S313", "kind": "iteration", "L": 100, "p": 32, "S": 313, "start": 1,
         "resume": 0, "ordered": 0, "trace": 0},
        # the headline configuration (16384 chains, L = 32) with the round cut from 10^5 sweeps; still too
        # large for the round record, as the whole one is
        {"name": "job_L32_p16384_S1000", "kind": "iteration", "L": 32, "p": 16384, "S": 1000, "start": 1,
         "resume": 1, "ordered": 0, "trace": 0},
        # the two larger configurations with their rounds cut: replayed joint, and recorded joint with the
        # per-sweep energy trace
        {"name": "job_L64_p4096_S1000", "kind": "iteration", "L": 64, "p": 4096, "S": 1000, "start": 1,
         "resume": 1, "ordered": 0, "trace": 0},
        {"name": "job_L128_p1024_S200", "kind": "iteration", "L": 128, "p": 1024, "S": 200, "start": 1,
         "resume": 0, "ordered": 0, "trace": 1},
        # the uneven batch: five jobs of different L per launch, two iterations in one CUDA graph
        {"name": "batch_uneven_S200", "kind": "batch", "S": 200, "iterations": 2, "scale": 1},
        # serving: the first jobs of the Poisson stream arriving as one burst, cut to a few iterations each
        {"name": "serving_24jobs", "kind": "serving", "jobs": 24, "iterations": 4, "S": 20, "slots": 16},
    ]


def _log_int(rng, lo, hi):
    return int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))


def draw(rng):
    kind = rng.choice(["iteration"] * 5 + ["attempts", "noalloc", "thermo", "batch", "serving"])
    if kind == "attempts":
        L = 4 * rng.randint(2, 16)
        return {"kind": kind, "L": L, "p": _log_int(rng, 8, 128), "n": _log_int(rng, 20, L * L - 1), "resume": 1}
    if kind == "thermo":
        return {"kind": kind, "L": 4 * rng.randint(2, 32), "betas": _log_int(rng, 1, 2000)}
    if kind == "batch":
        return {"kind": kind, "S": _log_int(rng, 10, 200), "iterations": rng.randint(1, 2), "scale": rng.randint(1, 8)}
    if kind == "serving":
        return {"kind": kind, "jobs": rng.randint(1, 24), "iterations": rng.randint(1, 4),
                "S": rng.randint(4, 20), "slots": rng.choice([4, 16, 32])}
    # generation: any L the library takes from 8 up, chains from a few dozen to 16384, rounds from one sweep
    # up, within 2.5e6 attempts a chain and 4e9 in all
    while True:
        L = 4 * rng.randint(2, 32)
        p = _log_int(rng, 32, 16384)
        S = _log_int(rng, 1, 5000)
        if S * L * L <= 2_500_000 and p * S * L * L <= 4_000_000_000:
            break
    if kind == "noalloc":
        return {"kind": kind, "L": L, "p": p, "S": S}
    return {"kind": kind, "L": L, "p": p, "S": S, "start": 1, "resume": rng.randint(0, 1),
            "ordered": 1 if rng.random() < 0.25 else 0, "trace": 1 if rng.random() < 0.25 else 0}


# ------------------------------------------------------------------ inputs
def _weights(L, rng):
    """A grown log-weight: -N H(m / N) with H the binary entropy (the slope of -ln g of the Ising
    model within a few percent over most of the range), plus the noise of an estimate."""
    N = L * L
    q = np.clip(np.arange(N + 1) / N, 1e-300, 1.0)
    r = np.clip(1.0 - np.arange(N + 1) / N, 1e-300, 1.0)
    return N * (q * np.log(q) + r * np.log(r)) + rng.normal(0.0, 0.05, N + 1)


def _pack(up):
    """bool [p][L][L] -> uint32 words [p][L][ceil(L / 32)], bit x % 32 of word x // 32."""
    p, L, _ = up.shape
    wd = (L + 31) // 32
    full = np.zeros((p, L, 32 * wd), np.uint8)
    full[:, :, :L] = up
    return np.ascontiguousarray(np.packbits(full, axis=2, bitorder="little")).view("<u4").reshape(p, L, wd)


def _spins(L, p, rng):
    """Chains spread over the energy range: every chain has its own share of up spins, and half of
    them are turned on one sublattice (the antiferromagnetic side)."""
    share = rng.uniform(0.5, 0.98, (p, 1, 1)).astype(np.float32)
    up = rng.random((p, L, L), dtype=np.float32) < share
    odd = (np.add.outer(np.arange(L), np.arange(L)) & 1).astype(bool)
    turned = rng.random((p, 1, 1)) < 0.5
    return up ^ (turned & odd[None])


def _levels(up):
    L = up.shape[1]
    s = np.where(up, 1, -1).astype(np.int32)
    E = -(s * (np.roll(s, -1, 1) + np.roll(s, -1, 2))).sum((1, 2))
    return (E + 2 * L * L) // 4


def _seed64(seed):
    return int(np.random.default_rng([7, seed]).integers(1, 1 << 62))


def _grown(case, seed):
    rng = np.random.default_rng([11, case["L"], seed])
    return _weights(case["L"], rng), _spins(case["L"], case["p"], rng)


def _visited_weights(case, seed):
    L = case["L"]
    rng = np.random.default_rng([13, L, seed])
    W = _weights(L, rng)
    vis = np.ones(L * L + 1, np.uint8)
    vis[1] = vis[L * L - 1] = 0          # these levels do not exist
    W[vis == 0] = 0.0
    return W, vis, np.linspace(0.05, 1.0, case["betas"])


def _batch_groups(case):
    return [(L, max(32, p // case["scale"]), s) for L, p, s in BATCH_GROUPS]


def _served(case):
    """(L, chains) of the burst: the first jobs of the serving stream."""
    return [(j.L, j.chains) for j in serving_stream(case["jobs"])]


# ------------------------------------------------------------------ prepare / run
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("iteration", "attempts"):
        job = mc.Job(case["L"], case["p"], _seed64(seed), case.get("start", 1))
        if case["resume"]:
            W, up = _grown(case, seed)
            job.weights = W
            job.spin_words = _pack(up)
        if case.get("ordered"):
            job.set_join_order(1)
        if case.get("trace"):
            job.set_trace(True)
        return {"case": case, "job": job}
    if kind == "noalloc":
        L, p = case["L"], case["p"]
        W, up = _grown(case, seed)
        return {"case": case, "seed": _seed64(seed), "t": 0,
                "spins": torch.from_numpy(_pack(up).view(np.int32)).cuda(),
                "levels": torch.from_numpy(_levels(up).astype(np.int32)).cuda(),
                "W": torch.from_numpy(W).cuda(),
                "hist": torch.zeros(L * L + 1, dtype=torch.int64, device="cuda")}
    if kind == "thermo":
        W, vis, betas = _visited_weights(case, seed)
        job = mc.Job(case["L"], 64, _seed64(seed), 1)
        job.weights = W
        job.visited = vis
        return {"case": case, "job": job, "betas": betas}
    if kind == "batch":
        jobs = [mc.Job(L, p, _seed64(seed) + s, 1) for L, p, s in _batch_groups(case)]
        mc.mc_batch_autotune(jobs, min(case["S"], 20))     # cached after the first: as a batch user's program does
        return {"case": case, "jobs": jobs}
    return {"case": case, "server": mc.Server(40 << 30, case["slots"]), "seed": _seed64(seed), "pass": 0}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "iteration":
        job = state["job"]
        job.run_sweeps(case["S"])
        kept = job.join()
        hist = job.hist
        job.update_weights()
        out = {"kept": kept, "hist": hist, "k": job.k, "offsets": job.offsets, "energies": job.energies,
               "spins": job.spin_words, "weights": job.weights}
        if case["trace"]:
            out["trace"] = job.trace
        return out
    if kind == "attempts":
        job = state["job"]
        job.run_attempts(case["n"])
        kept = job.join()
        return {"kept": kept, "hist": job.hist, "k": job.k, "energies": job.energies, "spins": job.spin_words}
    if kind == "noalloc":
        mc.mc_generate_noalloc(case["L"], case["p"], state["seed"], state["t"], case["S"],
                               state["spins"].data_ptr(), state["levels"].data_ptr(), state["W"].data_ptr(),
                               state["hist"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        state["t"] += case["S"] * case["L"] ** 2
        return {"spins": state["spins"], "levels": state["levels"], "hist": state["hist"]}
    if kind == "thermo":
        return state["job"].thermo(state["betas"])
    if kind == "batch":
        jobs = state["jobs"]
        mc.mc_batch_run(jobs, case["iterations"], case["S"], 2)
        return [{"weights": j.weights, "energies": j.energies, "spins": j.spin_words, "k": j.k} for j in jobs]
    srv = state["server"]
    ids = [srv.submit(L, p, state["seed"] + 100 * state["pass"] + i, case["iterations"], case["S"])
           for i, (L, p) in enumerate(_served(case))]
    state["pass"] += 1
    done = [srv.wait(i) for i in ids]
    return {"weights": np.concatenate([W for W, _ in done]),
            "joined": np.array([st["joined"] for _, st in done], np.int64),
            "attempts": np.array([st["attempts"] for _, st in done], np.int64)}


# ------------------------------------------------------------------ what a pass cannot do without
# integer operations of one attempt: its Philox word (a quarter of ten rounds of 2 multiplies and 2 xors),
# the aligned neighbours (7), the threshold (2), the compare (1), the flip (2), the level count (3); and of
# one sample's joint test: its Philox word, the threshold, the compare
OPS_ATTEMPT = 25
OPS_JOINT = 13


def _generation_work(L, p, attempts, kept_fraction_tested=1.0 / 64):
    N = L * L
    lat = 4 * p * L * ((L + 31) // 32)
    # lattices and levels in and out, the weight in, the histogram out
    return {"bytes": 2 * lat + 8 * p + 16 * (N + 1),
            "flops": p * attempts * (OPS_ATTEMPT + OPS_JOINT * kept_fraction_tested)}


def work(case):
    kind = case["kind"]
    if kind == "iteration":
        w = _generation_work(case["L"], case["p"], case["S"] * case["L"] ** 2)
        w["bytes"] += 16 * case["p"] + 8 * (case["L"] ** 2 + 1)            # k, offsets; the new weight
        if case["trace"]:
            w["bytes"] += 4 * case["p"] * case["S"]
        return w
    if kind == "attempts":
        return _generation_work(case["L"], case["p"], case["n"])
    if kind == "noalloc":
        return _generation_work(case["L"], case["p"], case["S"] * case["L"] ** 2, 0.0)
    if kind == "thermo":
        n = case["L"] ** 2 + 1
        # per level and beta: one exponential (~30 operations) and its three sums
        return {"bytes": 9 * n + 40 * case["betas"], "flops": 38 * n * case["betas"]}
    if kind == "batch":
        ws = [_generation_work(L, p, case["S"] * L * L) for L, p, _ in _batch_groups(case)]
    else:
        ws = [_generation_work(L, p, case["S"] * L * L) for L, p in _served(case)]
    return {q: case["iterations"] * sum(w[q] for w in ws) for q in ("bytes", "flops")}


# ------------------------------------------------------------------ the same in plain numpy
def _philox(blk, chain, w2, tag, seed):
    """Philox4x32-10 words [4][...] at counters (blk as 64 bits or (blk, w2), chain, tag)."""
    M0, M1 = np.uint64(0xD2511F53), np.uint64(0xCD9E8D57)
    lo = np.uint64(0xFFFFFFFF)
    chain = np.asarray(chain, np.uint64)
    c0 = np.full(chain.shape, blk & 0xFFFFFFFF, np.uint64) if np.isscalar(blk) else np.asarray(blk, np.uint64)
    c1 = np.full(chain.shape, w2, np.uint64)
    c2, c3 = chain.copy(), np.full(chain.shape, tag, np.uint64)
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        p0, p1 = M0 * c0, M1 * c2
        c0, c1, c2, c3 = ((p1 >> np.uint64(32)) ^ c1 ^ np.uint64(k0), p1 & lo,
                          (p0 >> np.uint64(32)) ^ c3 ^ np.uint64(k1), p0 & lo)
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return np.stack([c0, c1, c2, c3])


def _thresholds(d):
    """A 32-bit uniform u is accepted iff u <= ceil(2^32 e^d) - 1 (all of them for d >= 0, u = 0 for d <= -23)."""
    x = np.exp(np.clip(d, -23.0, 0.0)) * 4294967296.0
    t = np.where(x <= 1.0, 0.0, np.ceil(x) - 1.0)
    return np.where(d >= 0, 0xFFFFFFFF, np.where(d <= -23.0, 0, t)).astype(np.uint64)


def _generate(up, W, seed, n):
    """n typewriter attempts of every chain from the lattices `up` (changed in place): levels [n][p]."""
    p, L, _ = up.shape
    N = L * L
    m = _levels(up).astype(np.int64)
    idx = np.arange(N + 1)
    T = np.zeros((5, N + 1), np.uint64)
    for a in range(5):
        to = np.clip(idx + a - 2, 0, N)
        T[a] = _thresholds(W[to] - W[idx])
    lat = np.ascontiguousarray(up.reshape(p, N).T)        # [site][chain]
    chains = np.arange(p, dtype=np.uint64)
    out = np.zeros((n, p), np.int64)
    u = None
    for t in range(n):
        if t % 4 == 0:
            u = _philox(t >> 2, chains, 0, 0, seed)
        s = t % N
        y, x = divmod(s, L)
        c = lat[s]
        a = ((lat[y * L + (x - 1) % L] == c).astype(np.int64) + (lat[y * L + (x + 1) % L] == c) +
             (lat[((y - 1) % L) * L + x] == c) + (lat[((y + 1) % L) * L + x] == c))
        acc = u[t & 3] <= T[a, m]
        lat[s] = c ^ acc
        m = m + np.where(acc, a - 2, 0)
        out[t] = m
    up[:] = lat.T.reshape(p, L, L)
    return out


def _join(levels, W, seed, order):
    """The serial joint of a job's first round: k per chain, 0 where nothing is kept."""
    n, p = levels.shape
    k = np.zeros(p, np.int64)
    carry = None
    blocks = np.arange((n + 3) // 4, dtype=np.uint64)
    for c in order:
        if carry is None:
            k[c] = 1
        else:
            u = _philox(blocks, np.full(blocks.shape, int(c), np.uint64), 0, 1, seed)
            u = u.T.reshape(-1)[:n]
            hit = np.flatnonzero(u <= _thresholds(W[levels[:, c]] - W[carry]))
            if hit.size:
                k[c] = hit[0] + 1
        if k[c]:
            carry = levels[-1, c]
    return k


def _exact_round(case, seed, n):
    W, up = _grown(case, seed)
    levels = _generate(up, W, _seed64(seed), n)
    p, N = case["p"], case["L"] ** 2
    order = np.lexsort((np.arange(p), levels[-1])) if case.get("ordered") else np.arange(p)
    k = _join(levels, W, _seed64(seed), order)
    kept = np.where(k > 0, n - k + 1, 0)
    h = np.zeros(N + 1, np.int64)
    for c in range(p):
        if k[c]:
            h += np.bincount(levels[k[c] - 1:, c], minlength=N + 1)
    offsets = np.zeros(p, np.int64)
    offsets[order] = np.cumsum(kept[order]) - kept[order]
    return W, up, levels, k, kept, h, offsets


def exact(case, seed):
    kind = case["kind"]
    if kind == "thermo":
        W, vis, betas = _visited_weights(case, seed)
        N = case["L"] ** 2
        on = vis > 0
        W, E = W[on], (-2.0 * N + 4.0 * np.arange(N + 1))[on]
        out = np.zeros((betas.size, 4))
        lng = -W
        norm = N * np.log(2.0) - (lng.max() + np.log(np.exp(lng - lng.max()).sum()))
        for i, b in enumerate(betas):
            x = lng - b * E
            w = np.exp(x - x.max())
            Z = w.sum()
            Eav = (E * w).sum() / Z
            F = -(norm + x.max() + np.log(Z)) / b
            out[i] = Eav, b * b * (((E - Eav) ** 2) * w).sum() / Z, F, b * (Eav - F)
        return out
    if kind not in ("iteration", "attempts", "noalloc") or not case.get("resume", 1):
        return None
    N = case["L"] ** 2
    n = case["n"] if kind == "attempts" else case["S"] * N
    if n > EXACT_ATTEMPTS or n * case["p"] > EXACT_SAMPLES:
        return None
    if kind == "noalloc":
        W, up = _grown(case, seed)
        levels = _generate(up, W, _seed64(seed), n)
        return {"spins": torch.from_numpy(_pack(up).view(np.int32).copy()),
                "levels": torch.from_numpy(levels[-1].astype(np.int32)),
                "hist": torch.from_numpy(np.bincount(levels.reshape(-1), minlength=N + 1).astype(np.int64))}
    W, up, levels, k, kept, h, offsets = _exact_round(case, seed, n)
    out = {"kept": int(kept.sum()), "hist": h, "k": k}
    if kind == "iteration":
        out["offsets"] = offsets
    out["energies"] = (4 * levels[-1] - 2 * N).astype(np.int32)
    out["spins"] = _pack(up)
    if kind == "iteration":
        out["weights"] = np.where(h > 0, W - np.log(np.maximum(h, 1)), W)
        if case["trace"]:
            out["trace"] = (4 * levels[N - 1::N] - 2 * N).astype(np.int32)
    return out
