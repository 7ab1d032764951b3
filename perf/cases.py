"""The workloads whose speed is followed on a GB300.

Each listed case is one piece of work a user has the library do through its
public entry points (``paper_1012_0385_gb300.asep``): an ensemble run (re-draw
the initial lattices, advance, read the width table, the hop counters, the
other observables switched on and the lattices), a few sweeps of a running
context with its read-out, or one step of a batch of many contexts.  Sizes are
those of the benchmark's configurations and windows (``bench.py``) and of the
tests; ``draw`` spreads them over the ranges the library is used in.

All outputs are whole numbers except W^2 (one rounding of an exact ratio).
"""
from __future__ import annotations

import math
from decimal import Decimal, getcontext
from fractions import Fraction

import numpy as np

from paper_1012_0385_gb300 import asep as A
from paper_1012_0385_gb300.sampling import every, log_times

RING, TWO = "ring", "two_lane"
SCHED = {"domain": A.ASEP_SCHED_DOMAIN, "serial": A.ASEP_SCHED_SERIAL, "sca": A.ASEP_SCHED_SCA}
DIS = {"none": A.ASEP_DIS_NONE, "bimodal": A.ASEP_DIS_BIMODAL, "turning": A.ASEP_DIS_TURNING,
       "bimodal_pq": A.ASEP_DIS_BIMODAL_PQ, "crossing": A.ASEP_DIS_CROSSING}


def ensemble(name, schedule, L, samples, sweeps, **kw):
    """A case of one context: `realizations` x `samples` lattices of L sites per lane, `sweeps` sweeps a pass."""
    case = {"kind": "ensemble", "schedule": schedule, "model": RING, "L": L, "D": 0, "realizations": 1,
            "samples": samples, "sweeps": sweeps, "p": 1.0, "q": 0.0, "dis": "none", "dis_a": 0.0, "dis_b": 0.0,
            "dis_c": 0.0, "half_filling": False, "times": "end", "counts": True, "observables": False,
            "balance": 0}
    case.update(kw)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # The smallest calls, where launches and read-outs count: eight short rings, four sweeps, a record of each.
        ensemble("small_rings", "domain", 4096, 8, 4, D=256, times="each"),
        # Plain TASEP under exact serial random-sequential update, eight samples, a snapshot every 100 sweeps.
        ensemble("serial_plain_tasep", "serial", 4096, 8, 1000, times="every100"),
        # The serial reference as statistics use it: many rings at once (an odd number of them).
        ensemble("serial_many_rings", "serial", 4096, 2021, 100, p=0.75, q=0.25),
        # The growth regime, the headline workload (window of its 2^14 sweeps): W(t) at the log times, hop
        # counters off, balanced launches as the autotuner chooses them.
        ensemble("growth_rings", "domain", 1 << 17, 256, 2048, D=256, p=0.75, q=0.25, times="log", counts=False,
                 balance=16),
        # Quenched bimodal disorder (Q-TASEP), 64 realizations x 4 samples.
        ensemble("bimodal_rings", "domain", 1 << 16, 4, 1000, D=256, realizations=64, dis="bimodal", dis_a=0.1,
                 dis_b=0.3, times="log"),
        # The two-lane model with turning sites: currents, profile and autocorrelation recorded.
        ensemble("two_lane_turning", "domain", 1 << 16, 128, 1000, model=TWO, D=128, q=1.0, dis="turning", dis_a=0.05,
                 dis_b=0.1, half_filling=True, times="log", observables=True),
        # One step of the served mix: contexts of every family and uneven size in one persistent batch.
        {"name": "served_mix", "kind": "mix", "contexts": 24, "log2_L_max": 22, "samples_max": 48, "work": 1 << 27},
        # Rings beyond on-chip memory under the domain schedule: tiles streamed through shared memory.
        ensemble("streamed_rings", "domain", 1 << 24, 16, 60, D=256, p=0.75, q=0.25, counts=False),
        # The growth regime under the paper's own schedule (two-sub-lattice cellular automaton).
        ensemble("sca_growth_rings", "sca", 1 << 17, 256, 2048, p=0.75, q=0.25, times="log", counts=False),
        # The paper's two-lane sequence, in-lane rate 1/2, lane changes at turning sites.
        ensemble("sca_two_lane", "sca", 1 << 16, 128, 1000, model=TWO, p=0.5, q=0.5, dis="turning", dis_a=0.05,
                 dis_b=0.1, half_filling=True, times="log", observables=True),
        # Q-SSEP: independent slow classes for both hop directions, the paper's rates; a ragged ring (391 units).
        ensemble("sca_qssep", "sca", 256 * 391, 1, 1000, realizations=201, p=0.8, q=0.8, dis="bimodal_pq", dis_a=0.5,
                 dis_b=0.16, dis_c=0.16, times="log"),
        # The paper's one-large-sample mode: rings of 2^28 sites in device memory.
        ensemble("sca_streamed_rings", "sca", 1 << 28, 8, 800, p=0.75, q=0.25, counts=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sweeps(rng, lanes_sites, rate, least=1, most=4000, lo=3e-3, hi=60e-3):
    """Sweeps that take between `lo` and `hi` seconds at `rate` attempts/s."""
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(least, min(most, int(t * rate / lanes_sites)))


def draw(rng):
    """One more case: a family uniformly, its sizes over the whole range (ragged ones among them)."""
    fam = rng.choice(["small", "serial_few", "serial_many", "growth", "bimodal", "two_lane", "mix", "streamed", "sca",
                      "sca_two_lane", "sca_disorder", "sca_streamed"])
    rates = rng.choice([(1.0, 0.0), (0.75, 0.25), (0.8, 0.2), (0.5, 0.5), (0.6, 0.1)])
    times = rng.choice(["end", "log", "every100"])
    counts = rng.random() < 0.5
    if fam == "small":  # a short run, or a running context watched every few sweeps
        D, kind = rng.choice([32, 64, 128, 256]), rng.choice(["ensemble", "step"])
        return ensemble(None, "domain", 2 * D * _log(rng, 1, 24), _log(rng, 1, 64), rng.randint(2, 8), kind=kind,
                        D=D, p=rates[0], q=rates[1], times="each" if kind == "ensemble" else "none", counts=counts)
    if fam == "serial_few":
        L, S = 1 << rng.randint(7, 14), _log(rng, 1, 200)
        return ensemble(None, "serial", L, S, _sweeps(rng, L * S, 2.8e8 * min(S, 152)), p=rates[0], q=rates[1],
                        times=times, counts=counts)
    if fam == "serial_many":
        L, S = 1 << rng.randint(8, 16), _log(rng, 650, 3000)
        return ensemble(None, "serial", L, S, _sweeps(rng, L * S, 4e10), p=rates[0], q=rates[1], counts=counts)
    if fam == "growth":
        L, S = 512 * _log(rng, 40, 1000), _log(rng, 100, 500)
        return ensemble(None, "domain", L, S, _sweeps(rng, L * S, 5e11), D=256, p=rates[0], q=rates[1], times=times,
                        counts=counts, balance=rng.choice([0, 16, 32]))
    if fam == "bimodal":
        L, R, S = 512 * _log(rng, 24, 400), _log(rng, 16, 120), rng.randint(1, 4)
        return ensemble(None, "domain", L, S, _sweeps(rng, L * R * S, 2e11), D=256, realizations=R, p=rates[0],
                        q=rates[1], dis=rng.choice(["bimodal", "bimodal_pq"]), dis_a=rng.choice([0.1, 0.5]),
                        dis_b=0.3, dis_c=0.1 if rates[1] else 0.0, times=times, counts=counts)
    if fam == "two_lane":
        L, S = 256 * _log(rng, 32, 400), _log(rng, 60, 300)
        return ensemble(None, "domain", L, S, _sweeps(rng, 2 * L * S, 2e11), model=TWO, D=128, q=1.0, dis="turning",
                        dis_a=rng.choice([0.05, 0.1, 0.2]), dis_b=0.1, half_filling=True, times=times,
                        observables=rng.random() < 0.5)
    if fam == "mix":
        return {"kind": "mix", "contexts": rng.randint(4, 40), "log2_L_max": rng.randint(14, 22),
                "samples_max": _log(rng, 4, 64), "work": 1 << rng.randint(22, 27)}
    if fam == "streamed":
        L, S = (1 << 24) + 512 * _log(rng, 1, 1 << 16), rng.randint(1, 10)
        return ensemble(None, "domain", L, S, _sweeps(rng, L * S, 5e11), D=256, p=rates[0], q=rates[1], counts=counts)
    if fam == "sca":
        L, S = 256 * _log(rng, 9, 2000), _log(rng, 40, 400)
        return ensemble(None, "sca", L, S, _sweeps(rng, L * S, 4e12), p=rates[0], q=rates[1], times=times,
                        counts=counts)
    if fam == "sca_two_lane":
        L, S = 256 * _log(rng, 24, 800), _log(rng, 40, 300)
        return ensemble(None, "sca", L, S, _sweeps(rng, 2 * L * S, 1e12), model=TWO, p=0.5, q=0.5,
                        dis=rng.choice(["none", "turning", "turning"]), dis_a=rng.choice([0.05, 0.1]), dis_b=0.1,
                        half_filling=True, times=times, observables=rng.random() < 0.5)
    if fam == "sca_disorder":
        L, R = 256 * _log(rng, 24, 800), _log(rng, 60, 400)
        return ensemble(None, "sca", L, 1, _sweeps(rng, L * R, 1.2e12), realizations=R, p=0.8,
                        q=rng.choice([0.0, 0.8]), dis=rng.choice(["bimodal", "bimodal_pq"]), dis_a=0.5, dis_b=0.16,
                        dis_c=0.16, times=times, counts=counts)
    L, S = 256 * _log(rng, 5800, 1 << 19), rng.randint(1, 8)
    return ensemble(None, "sca", L, S, _sweeps(rng, L * S, 5e12), p=rates[0], q=rates[1], counts=counts)


def _times(case):
    n, kind = case["sweeps"], case["times"]
    if kind == "none":
        return []
    t = {"end": [0], "each": every(1, n), "log": log_times(n), "every100": every(100, n)}[kind]
    return sorted(set(t) | {n})


def _params(case, seed):
    th = A.asep_threshold
    flags = 0 if case["counts"] or case["model"] == TWO else A.ASEP_FLAG_NO_HOP_COUNTS
    kw = dict(model=A.ASEP_MODEL_TWO_LANE if case["model"] == TWO else A.ASEP_MODEL_RING,
              schedule=SCHED[case["schedule"]], L=case["L"], domain_sites=case["D"],
              n_realizations=case["realizations"], samples_per_real=case["samples"], p_thr=th(case["p"]),
              q_thr=th(case["q"]), dis_kind=DIS[case["dis"]], dis_a_thr=th(case["dis_a"]),
              dis_b_thr=th(case["dis_b"]), dis_c_thr=th(case["dis_c"]), dis_seed=seed + 2, seed=seed + 1,
              init_kind=A.ASEP_INIT_BERNOULLI_HALF if case["half_filling"] else A.ASEP_INIT_FLAT_ALT,
              init_seed=seed + 4)
    times = _times(case)
    if case["observables"] and times:
        flags |= A.ASEP_FLAG_PROFILE | A.ASEP_FLAG_AUTOCORR
        kw["autocorr_t0"] = min(t for t in times if 2 * t >= case["sweeps"])
    return A.make_params(flags=flags, **kw), times


def _mix_jobs(case, seed):
    """The contexts of a served mix: the four workload families, L log-uniform from 2^10 up, samples log-uniform;
    each advances by the sweeps that come nearest to `work` attempts.  The sizes are the case's, the seeds differ."""
    rng = np.random.default_rng([17, case["contexts"], case["log2_L_max"], case["samples_max"]])
    jobs = []
    for k in range(case["contexts"]):
        fam = ["tasep", "asep", "bimodal", "two_lane"][k % 4]
        D = 128 if fam == "two_lane" else 256
        L = max(1, int(2 ** rng.uniform(10, case["log2_L_max"])) // (2 * D)) * 2 * D
        if L > 1 << 18:
            L = L // 4096 * 4096  # rings spread over several CTAs: a multiple of 128 words
        S = int(round(math.exp(rng.uniform(0, math.log(case["samples_max"])))))
        S = max(1, min(S, (1 << 23) // L))
        lanes = 2 if fam == "two_lane" else 1
        n = max(1, min(64, case["work"] // (lanes * L * S)))
        kw = {"tasep": {}, "asep": {"p": 0.75, "q": 0.25}, "bimodal": {"dis": "bimodal", "dis_a": 0.1, "dis_b": 0.3},
              "two_lane": {"model": TWO, "q": 1.0, "dis": "turning", "dis_a": 0.05, "dis_b": 0.1,
                           "half_filling": True}}[fam]
        jobs.append((ensemble(None, "domain", L, S, n, D=D, **kw), seed + 1000 * k))
    return jobs


def prepare(case, seed):
    if case["kind"] == "mix":
        jobs = _mix_jobs(case, seed)
        ctxs = [A.asep_create(*_params(c, s)) for c, s in jobs]
        batch = A.asep_batch_create(max_jobs=len(jobs), max_items=1 << 14)
        return {"case": case, "ctxs": ctxs, "n": [c["sweeps"] for c, _ in jobs], "batch": batch, "seed": seed}
    ctx = A.asep_create(*_params(case, seed))
    if case["balance"]:
        A.asep_set_balance(ctx, case["balance"])
    return {"case": case, "ctx": ctx, "seed": seed}


def _width(ctx):
    sum_h, sum_h2, w2 = A.asep_width(ctx)
    return {"sum_h": sum_h, "sum_h2": sum_h2.view(np.int64), "w2": w2}


def run(state):
    case = state["case"]
    if case["kind"] == "mix":
        A.asep_batch_sweep(state["batch"], state["ctxs"], state["n"])
        out = []
        for ctx in state["ctxs"]:
            out += [A.asep_counters(ctx).view(np.int64), _flat_states([ctx])]
        # the harness takes at most 64 arrays: the contexts' counters and lattices, each as one array
        return {"counters": np.concatenate(out[0::2]), "lattices": np.concatenate(out[1::2])}
    ctx = state["ctx"]
    if case["kind"] == "step":
        A.asep_sweep(ctx, case["sweeps"])
        return {"counters": A.asep_counters(ctx).view(np.int64), "lattices": _flat_states([ctx])}
    A.asep_reset(ctx, seed=state["seed"] + 1, init_seed=state["seed"] + 4)
    A.asep_sweep(ctx, case["sweeps"])
    out = _width(ctx)
    if case["counts"] or case["model"] == TWO:
        out["currents"] = A.asep_currents(ctx)
    if case["observables"]:
        out["profile"] = A.asep_profile(ctx).view(np.int32)
        out["autocorr"] = A.asep_autocorr(ctx)
    out["lattices"] = _flat_states([ctx])
    return out


def _flat_states(ctxs):
    return np.concatenate([A.asep_state(c)[0].reshape(-1) for c in ctxs]).view(np.int32) if len(ctxs) > 1 else \
        A.asep_state(ctxs[0])[0].reshape(-1).view(np.int32)


def work(case):
    """Bytes: the lattices and quenched planes read once, the lattices and tables written once.  "flops" are 32-bit
    integer operations: 24 an attempt for the random-sequential schedules (a quarter of a Philox4x32-10 call = 10, the
    update 14), and for the bit-sliced automaton (13 K + 12) / 32 with K random planes (those a threshold needs, at
    most the seven that decide all 64 candidate bonds of a thread on average)."""
    if case["kind"] == "mix":
        parts = [work(c) for c, _ in _mix_jobs(case, 0)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    lanes = 2 if case["model"] == TWO else 1
    planes = {"none": 0, "bimodal": 1, "turning": 1, "bimodal_pq": 2, "crossing": 2}[case["dis"]]
    S = case["realizations"] * case["samples"]
    words = case["L"] // 32
    attempts = lanes * case["L"] * S * case["sweeps"]
    if case["schedule"] == "sca":
        need = [0]
        for r in (case["p"], case["q"], case["dis_b"], case["dis_c"]):
            t = A.asep_threshold(r) >> 12
            if 0.0 < r < 1.0:
                need.append(20 - ((t & -t).bit_length() - 1))
        ops = (13 * min(7, max(need)) + 12) / 32
    else:
        ops = 24
    table = len(_times(case)) * S * lanes * 24
    return {"bytes": 4 * words * (2 * S * lanes + planes * case["realizations"]) + table, "flops": ops * attempts}


# ---------------------------------------------------------------------------
# Reference in plain numpy: rings without disorder under the domain schedule
# ---------------------------------------------------------------------------

def _philox(c, seed):
    """Philox4x32-10 of arrays of four counter words (Salmon, Moraes, Dror, Shaw, SC'11)."""
    m32 = np.uint64(0xFFFFFFFF)
    x, y, z, w = (np.asarray(v, dtype=np.uint64) & m32 for v in np.broadcast_arrays(*c))
    kx, ky = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * x, np.uint64(0xCD9E8D57) * z
        x, y, z, w = ((b >> np.uint64(32)) ^ y ^ np.uint64(kx), b & m32, (a >> np.uint64(32)) ^ w ^ np.uint64(ky), a & m32)
        kx, ky = (kx + 0x9E3779B9) & 0xFFFFFFFF, (ky + 0xBB67AE85) & 0xFFFFFFFF
    return x, y, z, w


def _poisson(m):
    """floor(2^32 P(Poisson(m) <= k)) for k = 0, 1, ... up to the first 2^32 - 1."""
    getcontext().prec = 80
    term, acc, out, k = (-Decimal(m)).exp(), Decimal(0), [], 0
    while True:
        acc += term
        t = int((acc * (1 << 32)).to_integral_value(rounding="ROUND_FLOOR"))
        if t >= (1 << 32) - 1:
            return np.array(out, dtype=np.uint64)
        out.append(t)
        k += 1
        term = term * m / k


def exact(case, seed):
    """W^2 of a short run of rings without disorder, replayed in numpy from the definition of the domain schedule;
    None for whole numbers (lattices, sums, counters) and for longer runs."""
    if case["kind"] != "ensemble" or case["schedule"] != "domain" or case["model"] != RING or case["dis"] != "none":
        return None
    L, S, n = case["L"], case["samples"], case["sweeps"]
    D = case["D"] or 256
    if not case["D"]:
        while D > 32 and L % (2 * D):
            D //= 2
    if S * (L // D) * n > 4e6 or 300 * n > 60000 or case["half_filling"]:
        return None
    th = lambda p: 0xFFFFFFFF if p >= 1 else math.floor(p * 1048576 + 0.5) << 12  # noqa: E731
    pt, qt = th(case["p"]), th(case["q"])
    acc = lambda r, t: (r & np.uint64(0xFFFFF000)) < np.uint64(t) if t != 0xFFFFFFFF else np.ones(r.shape, bool)  # noqa: E731
    tab, G, key = _poisson(D), L // (2 * D), seed + 1
    sites = np.tile((np.arange(L) % 2 == 0).astype(np.int8), (S, 1))
    sample, times, w2 = np.arange(S), _times(case), []
    rows = sample[:, None]

    def record():
        h = np.cumsum(2 * sites.astype(np.int64) - 1, axis=1)
        w2.append([[float(Fraction(L * int((r * r).sum()) - int(r.sum()) ** 2, L * L))] for r in h])

    if 0 in times:
        record()
    for s in range(n):
        off = (_philox((s, 3 << 8, sample, 0), key)[0] & np.uint64(2 * D - 1)).astype(np.int64)
        for phase in (0, 1):
            dom = 2 * np.arange(G) + phase
            start = (off[:, None] + D * dom[None, :]) % L
            words = list(_philox((s, 4 << 8, rows, dom[None, :]), key))
            K = np.searchsorted(tab, words[0], side="right")
            for k in range(1, int(K.max()) + 1):
                if k % 4 == 0:
                    words = list(_philox((s, (4 << 8) | ((k // 4) << 12), rows, dom[None, :]), key))
                r = words[k % 4]
                i = (start + (r & np.uint64(D - 1)).astype(np.int64)) % L
                j = (i + 1) % L
                a, b = sites[rows, i], sites[rows, j]
                hop = (k <= K) & (((a == 1) & (b == 0) & acc(r, pt)) | ((a == 0) & (b == 1) & acc(r, qt)))
                sites[np.broadcast_to(rows, hop.shape)[hop], i[hop]] ^= 1
                sites[np.broadcast_to(rows, hop.shape)[hop], j[hop]] ^= 1
        if s + 1 in times:
            record()
    out = {"sum_h": None, "sum_h2": None, "w2": np.array(w2), "lattices": None}
    if case["counts"]:
        out["currents"] = None
    return out
