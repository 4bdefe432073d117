"""The work that programs built on this library have it do, as cases that can be timed.

Sizes and schedules are those of this repository's workloads and studies (``bench.py``,
``instances.py``): the N = 16 latency case, the time-to-solution sizes (256 replicas,
n = 8..1024), the N = 200 dense workload, the N = 2000 complete graph, batches of uneven
sparse instances, serving streams; and odd sizes between them.  A case is prepared once (an
instance on the device, a handle or a batch, a schedule) and run any number of times; a run
starts from the same seed each time, so that its results are the same ones.

Kinds: ``anneal`` (a whole run and every replica's record), ``chunk`` (iterations
[t0, t0 + steps) of a longer run from states that the caller holds, resumable), ``csr`` (one
sparse instance), ``batch`` (many instances of uneven size together), ``serve`` (a burst of
requests through the continuous-batching server).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2407_10205_gb300 import instances as ins
from paper_2407_10205_gb300 import phia


def listed():
    return [
        # One replica of the 16-spin SK instance: the time of an iteration and nothing else.
        dict(name="sk16-single", kind="anneal", n=16, kmax=1, hmax=0, frac_bits=0, replicas=1, steps=1000, refresh=0),
        # The time-to-solution study's ordinary sizes: 256 replicas, couplings {-1, +1}.
        dict(name="tts-sk64", kind="anneal", n=64, kmax=1, hmax=0, frac_bits=0, replicas=256, steps=1000, refresh=50),
        # The N = 200 workload (integer couplings and fields in [-7, 7]).
        dict(name="dense200", kind="anneal", n=200, kmax=7, hmax=7, frac_bits=0, replicas=1024, steps=2000,
             refresh=50),
        # The study's largest size on one CTA with fixed-point couplings (7 fractional bits).
        dict(name="tts-spin256", kind="anneal", n=256, kmax=127, hmax=127, frac_bits=7, replicas=256, steps=2000,
             refresh=50),
        # A caller that holds the states and advances them in chunks; odd size, ragged count.
        dict(name="chunk333", kind="chunk", n=333, kmax=3, hmax=3, frac_bits=0, replicas=500, steps=200, total=2000,
             refresh=50),
        # The study past the on-chip sizes: few replicas, many short iterations.
        dict(name="tts-sk512", kind="anneal", n=512, kmax=1, hmax=0, frac_bits=0, replicas=256, steps=2000,
             refresh=50),
        # A few iterations at a time from states that the caller looks at in between;
        # fixed-point couplings, odd size.
        dict(name="chunk1001", kind="chunk", n=1001, kmax=127, hmax=127, frac_bits=7, replicas=600, steps=8,
             total=2000, refresh=50),
        # The complete graph of the default workload, on a handle that was autotuned for it.
        dict(name="sk2000", kind="anneal", n=2000, kmax=1, hmax=0, frac_bits=0, replicas=4096, steps=500, refresh=50,
             tune=1),
        # A serving request for a large dense instance: one chunk of 200 iterations.
        dict(name="serve-chunk6000", kind="chunk", n=6000, kmax=1, hmax=0, frac_bits=0, replicas=256, steps=200,
             total=5000, refresh=50),
        # A serving request for a large sparse instance (8 fractional bits, density 0.01).
        dict(name="sparse5000", kind="csr", n=5000, density=0.01, kmax=127, hmax=127, frac_bits=8, replicas=256,
             steps=400, refresh=50),
        # Uneven instances annealed together: sparse ones of the batch workload's sizes and
        # small dense ones among them.
        dict(name="batch-mixed", kind="batch", sparse=48, dense=16, n_lo=100, n_hi=3000, replicas=256, steps=200,
             refresh=50),
        # Requests that arrive together at the server and run to their step cap.
        dict(name="serve-burst", kind="serve", requests=16, n_lo=64, n_hi=2048, replicas=256, steps=600, refresh=50),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["anneal", "anneal", "anneal", "large", "large", "chunk", "chunk", "csr", "batch"])
    kmax, hmax, frac = rng.choice([(1, 0, 0), (7, 7, 0), (127, 127, 7), (16, 31, 2)])
    refresh = rng.choice([0, 20, 50, 50])
    if kind == "anneal":       # the sizes of the resident kernels
        n = _log_int(rng, 8, 384)
        return dict(kind="anneal", n=n, kmax=kmax, hmax=hmax, frac_bits=frac, replicas=_log_int(rng, 1, 2048),
                    steps=_log_int(rng, 100, 2000), refresh=refresh)
    if kind == "large":
        n = _log_int(rng, 385, 4096)
        replicas = _log_int(rng, 32, 4096)
        cap = int(2.0e12 / (float(n) * n * replicas))          # field multiply-adds of the N = 2000 case: 8.2e12
        return dict(kind="anneal", n=n, kmax=kmax, hmax=hmax, frac_bits=frac, replicas=replicas,
                    steps=max(8, min(cap, _log_int(rng, 50, 1000))), refresh=refresh)
    if kind == "chunk":
        n = _log_int(rng, 100, 4096)
        replicas = _log_int(rng, 32, 2048)
        cap = int(2.0e12 / (float(n) * n * replicas))
        steps = max(4, min(cap, _log_int(rng, 4, 400)))
        return dict(kind="chunk", n=n, kmax=kmax, hmax=hmax, frac_bits=frac, replicas=replicas, steps=steps,
                    total=steps * rng.randint(1, 10), refresh=refresh)
    if kind == "csr":
        n = _log_int(rng, 64, 6000)
        return dict(kind="csr", n=n, density=round(rng.uniform(0.006, 0.06), 4), kmax=127, hmax=rng.choice([31, 127]),
                    frac_bits=rng.choice([4, 8]), replicas=_log_int(rng, 16, 512), steps=_log_int(rng, 50, 400),
                    refresh=refresh)
    return dict(kind="batch", sparse=rng.randint(4, 40), dense=rng.randint(0, 24), n_lo=100,
                n_hi=_log_int(rng, 400, 3000), replicas=rng.choice([64, 200, 256]), steps=_log_int(rng, 50, 200),
                refresh=refresh)


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _dense(case, seed):
    """Couplings (int8, symmetric, zero diagonal) and fields (int32) on the device: k in
    {-1, +1} for kmax = 1, else uniform integers in [-kmax, kmax]."""
    n, g = case["n"], _gen(seed)
    if case["kmax"] == 1:
        u = torch.randint(0, 2, (n, n), generator=g, device="cuda", dtype=torch.int8) * 2 - 1
    else:
        u = torch.randint(-case["kmax"], case["kmax"] + 1, (n, n), generator=g, device="cuda", dtype=torch.int16)
        u = u.to(torch.int8)
    u = torch.triu(u, 1)
    k = (u + u.t()).contiguous()
    h = torch.randint(-case["hmax"], case["hmax"] + 1, (n,), generator=g, device="cuda", dtype=torch.int32)
    return k, h


def _beta1(n, kmax, frac_bits, degree):
    """The end of the linear schedule: a typical potential jump of 6 max(1, sqrt(n / 128))."""
    rms = 1.0 if kmax == 1 else math.sqrt(kmax * (kmax + 1) / 3.0)
    return 6.0 * max(1.0, math.sqrt(n / 128.0)) / (math.ldexp(rms, -frac_bits) * math.sqrt(max(degree, 1.0)))


def _schedule(case, degree=None):
    b1 = _beta1(case["n"], case["kmax"], case["frac_bits"], case["n"] - 1 if degree is None else degree)
    return phia.schedule(b1 / 20.0, b1, 0.1, 2.0, refresh=case["refresh"])


def _states(case, seed):
    g = _gen(seed + 1)
    shape = (case["replicas"], case["n"])
    return (torch.randn(shape, generator=g, device="cuda"), torch.randn(shape, generator=g, device="cuda"))


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": seed}
    if kind in ("anneal", "chunk"):
        k, h = _dense(case, seed)
        st["sched"] = _schedule(case)
        st["annealer"] = phia.Annealer(k, h, case["frac_bits"])
        if case.get("tune"):
            phia.autotune(st["annealer"].h, st["sched"], case["replicas"], probe_iters=60)
        if kind == "chunk":
            st["x0"], st["v0"] = _states(case, seed)
            st["x"], st["v"] = torch.empty_like(st["x0"]), torch.empty_like(st["v0"])
    elif kind == "csr":
        c = ins.erdos_renyi(case["n"], case["density"], case["kmax"], case["hmax"], case["frac_bits"], seed)
        st["sched"] = _schedule(case, degree=case["density"] * case["n"])
        st["annealer"] = phia.Annealer(h_k=c.kh, frac_bits=c.frac_bits, csr=(c.row_ptr, c.col, c.val))
    elif kind == "batch":
        rng = random.Random(case["sparse"] + 1000 * case["dense"])     # the sizes belong to the case
        members = [ins.erdos_renyi(rng.randint(case["n_lo"], case["n_hi"]), rng.uniform(0.006, 0.06), 127, 31, 4,
                                   1000 * seed + q) for q in range(case["sparse"])]
        for q in range(case["dense"]):
            members.insert(rng.randint(0, len(members)), ins.dense_int(_log_int(rng, 64, 384), 7, 7, 1000 * seed + q))
        st["sched"] = phia.schedule(0.01, 0.18, 0.1, 2.0, refresh=case["refresh"])
        st["batch"] = phia.Batch(members)
        st["count"] = len(members)
    else:
        rng = random.Random(case["requests"])                          # the sizes belong to the case
        st["requests"] = []
        for q in range(case["requests"]):
            n = _log_int(rng, case["n_lo"], case["n_hi"])
            if q % 2 == 0:
                inst, kmax, frac, degree = ins.sk_pm1(n, 1000 * seed + q), 1, 0, n - 1
            else:
                inst, kmax, frac, degree = ins.erdos_renyi(n, 0.01, 127, 127, 8, 1000 * seed + q), 127, 8, 0.01 * n
            b1 = _beta1(n, kmax, frac, degree)
            st["requests"].append((inst, phia.schedule(b1 / 20.0, b1, 0.1, 2.0, refresh=case["refresh"]), seed + q))
        st["server"] = phia.Server(max_inflight=16, hbm_budget_bytes=16 << 30, chunk_iters=200)
    return st


def run(state):
    case, seed = state["case"], state["seed"]
    kind, R, T = case["kind"], case["replicas"], case["steps"]
    if kind in ("anneal", "csr"):
        A = state["annealer"]
        res = A.anneal(state["sched"], R, T, seed)
        e, step, hit, bits = phia.replica_results(A.h, R, A.n)
        return {"energy": res.energy_k, "spins": res.spins, "best_e": e, "best_step": step, "hit": hit, "bits": bits}
    if kind == "chunk":
        A, x, v = state["annealer"], state["x"], state["v"]
        x.copy_(state["x0"])
        v.copy_(state["v0"])
        phia.run(A.h, state["sched"], R, 0, T, case["total"], seed, x, v)
        e, step, hit, bits = phia.replica_results(A.h, R, A.n)
        return {"x": x, "v": v, "best_e": e, "best_step": step, "hit": hit, "bits": bits}
    if kind == "batch":
        b = state["batch"]
        b.anneal(state["sched"], R, T, seed)
        best = [b.best(q) for q in range(state["count"])]
        recs = [b.replica_results(q, R) for q in range(state["count"])]
        return {"energy": np.array([e for e, _ in best], dtype=np.int64), "spins": np.concatenate([s for _, s in best]),
                "best_e": np.stack([r[0] for r in recs]), "best_step": np.stack([r[1] for r in recs]),
                "bits": np.concatenate([r[3].reshape(-1) for r in recs])}
    srv = state["server"]
    ids = [srv.submit(inst, sched, R, T, s) for inst, sched, s in state["requests"]]
    srv.wait_all()
    done = [srv.poll(i, want_spins=True) for i in ids]
    return {"energy": np.array([st.energy_k for st, _ in done], dtype=np.int64),
            "steps": np.array([st.steps_run for st, _ in done], dtype=np.int64),
            "spins": np.concatenate([s for _, s in done])}


# ------------------------------------------------------------------ what a run cannot do without

def work(case):
    """Field multiply-adds at 2 flops each and about 20 flops of update per spin, replica and
    iteration; couplings, fields and given states read once, records and states written once."""
    kind, R, T = case["kind"], case["replicas"], case["steps"]
    if kind in ("batch", "serve"):
        # expected sizes: sparse members uniform in [n_lo, n_hi] with mean density 0.033,
        # dense ones log-uniform in [64, 384]; requests log-uniform, half dense, half sparse
        if kind == "batch":
            lo, hi = case["n_lo"], case["n_hi"]
            n1, n2 = (lo + hi) / 2.0, (lo * lo + lo * hi + hi * hi) / 3.0
            spins, macs = case["sparse"] * n1, case["sparse"] * 0.033 * n2
            lo, hi, cnt, share = 64.0, 384.0, case["dense"], 1.0
        else:
            spins = macs = 0.0
            lo, hi, cnt, share = float(case["n_lo"]), float(case["n_hi"]), case["requests"], 0.505
        ln = math.log(hi / lo)
        spins += cnt * (hi - lo) / ln
        macs += cnt * share * (hi * hi - lo * lo) / (2.0 * ln)
        return {"bytes": 5.0 * macs + 4.0 * spins + R * spins / 8.0, "flops": R * T * (2.0 * macs + 20.0 * spins)}
    n = case["n"]
    macs = n * n * (case["density"] if kind == "csr" else 1.0)
    byts = macs * (5.0 if kind == "csr" else 1.0) + 4.0 * n + R * (24.0 + n / 8.0)
    if kind == "chunk":
        byts += 16.0 * R * n
    return {"bytes": byts, "flops": R * T * (2.0 * macs + 20.0 * n)}


# ------------------------------------------------------------------ in 64 bits

def exact(case, seed):
    """The states after a few iterations in FP64.  After many, a position that rounds to the
    other side of 0 has sent its replica another way, so longer runs have no such value; the
    records are whole numbers."""
    if case["kind"] != "chunk" or case["steps"] > 8 or 0 < case["refresh"] < case["steps"]:
        return None
    k, h = _dense(case, seed)
    x, v = (s.double() for s in _states(case, seed))
    sched, q = _schedule(case), math.ldexp(1.0, -case["frac_bits"])
    J, hq = k.double(), h.double()
    for t in range(case["steps"]):
        x = x + sched.eps * v
        s = torch.where(x >= 0, 1.0, -1.0).double()
        field = (s @ J + hq) * q
        beta = sched.beta0 + (sched.beta1 - sched.beta0) * (t / max(case["total"] - 1, 1))
        y = torch.tanh(sched.gamma * x)
        v = v + sched.eps * (beta * sched.gamma * (1.0 - y * y) * field - x)
    return {"x": x, "v": v, "best_e": None, "best_step": None, "hit": None, "bits": None}
