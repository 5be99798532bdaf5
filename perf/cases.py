"""The calls whose speed matters to a user of the plan evaluator, over the range of sizes that they take.

A user holds one planning window (a problem), a context made for it, and batches of candidate plans; each pass is the call such a
user makes on a batch.  `kind` says which:

  step         forecast, evaluation and top-k of a device-resident batch (a scheduler's tick)
  host         the same step from and to page-locked host memory, every plan's metrics returned
  phi          evaluation with the window terms of Eq. 12 and the top-k by that key
  next_use     evaluation under reclamation by next use, and top-k
  batch        evaluation under the replica batch limit B_q, and top-k
  stochastic   evaluation with S latency samples a plan, and top-k
  construct    plans built by the list scheduler
  search       one round of local search (children of the k best plans, their evaluation, the merge)
  static       evaluation without a context or any allocation (a scheduler inside a serving engine)

Windows are made of the repository's three workflow families (repair chains, fan-out / fan-in, random layers) with lognormal run
times; plans have uniform placements over the devices that fit, random topological dispatch orders and random bits.  All is drawn
from the seed, the plans on the GPU.  Every output is a whole number, and another correct implementation gives the same ones.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2609_03335_gb300 import wf

DEV = "cuda"
GIB = 1024  # MiB
# Device classes (capacity GiB, run-time multiplier, load GB/s) and model weights (GiB); a window takes a spread of each.
CLASSES = ((24, 1.0, 3), (48, 0.6, 6), (80, 0.4, 10), (141, 0.3, 10))
WEIGHTS = (3, 70, 14, 28, 6, 40, 16, 8, 4, 64, 20, 32, 10, 24, 12, 48)
STATIC_BYTES = 32 << 20  # the static entry point's scratch

# Fields of a case that most cases leave at these values.
DEFAULTS = dict(gap_ms=500, retain=False, grant=0, margin=0, bad=0.0, S=0, B=0, jitter=0, n_ops=0)


def _case(name, kind, N, W, D, M, P, k, **more):
    c = dict(DEFAULTS, kind=kind, N=N, W=W, D=D, M=M, P=P, k=k, **more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # One small workflow planned interactively: latency and launches count.
        _case("tiny_step", "step", 12, 1, 3, 4, 1024, 8),
        # A tick over a mix of 16 workflows that arrive together: many short plans.
        _case("mix_step", "step", 169, 16, 8, 6, 65536, 32, gap_ms=0),
        # The headline: a burst of 64 sessions.
        _case("burst_step", "step", 2000, 64, 8, 8, 16384, 32),
        # The same window planned by a process whose plans live in host memory; a ragged batch.
        _case("burst_host", "host", 2000, 64, 8, 8, 15001, 32),
        # A large pool and window; its times run past 32 bits.
        _case("large_step", "step", 8192, 256, 16, 12, 131072, 64),
        # Odd sizes, every option at once: retain rows, grants, a memory margin, some invalid plans, the window key.
        _case("ragged_phi", "phi", 1001, 37, 5, 11, 5003, 100, retain=True, grant=1500, margin=256, bad=0.02),
        # The burst under the paper's preferred reclamation order.
        _case("burst_next_use", "next_use", 2000, 64, 8, 8, 16384, 32),
        # The burst on replicas that batch up to four units.
        _case("burst_batch4", "batch", 2000, 64, 8, 8, 16384, 32, B=4),
        # Robust planning: 64 latency samples a plan.
        _case("stochastic_step", "stochastic", 500, 16, 8, 8, 8192, 32, S=64),
        # A fresh batch of good plans for the burst.
        _case("burst_construct", "construct", 2000, 64, 8, 8, 16384, 32, jitter=200_000),
        # One round of search around the 32 best plans of the burst.
        _case("burst_search", "search", 2000, 64, 8, 8, 16352, 32, n_ops=3),
        # The burst scored inside a serving engine that has no memory to give.
        _case("burst_static", "static", 2000, 64, 8, 8, 1900, 32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "host", "phi", "next_use", "batch", "stochastic", "construct", "search", "static"))
    # plan-positions (samples counted) that keep a pass below the largest listed case's
    most = {"step": 1 << 29, "host": 1 << 26, "stochastic": 1 << 28, "static": 1 << 22}.get(kind, 1 << 25)
    N = _log(rng, 12, 1000 if kind == "stochastic" else 8192 if kind == "step" else 3000)
    W = max(1, min(N // 4, round(N / rng.uniform(8, 40))))
    D, M = rng.randint(2, 16), rng.randint(2, 12)
    S = _log(rng, 8, 200) if kind == "stochastic" else 0
    P = _log(rng, 64, max(64, min(131072, most // (N * max(1, S)))))
    if kind == "static":
        P = min(P, _static_plans(N, W, D, M))
    B = rng.randint(1, 8) if kind == "batch" else 0
    return _case(None, kind, N, W, D, M, P, min(P, rng.choice((1, 8, 32, 64, 250))), gap_ms=rng.choice((0, 100, 500)),
                 retain=kind not in ("batch", "construct") and rng.random() < 0.3, grant=rng.choice((0, 0, 1500)),
                 margin=0 if kind == "static" else rng.choice((0, 0, 256)),
                 bad=rng.choice((0.0, 0.02)) if kind not in ("construct", "search") else 0.0, S=S, B=B,
                 jitter=rng.choice((0, 50_000, 200_000)) if kind == "construct" else 0,
                 n_ops=rng.randint(1, 8) if kind == "search" else 0)


def _static_plans(N, W, D, M):
    """The most plans of such a window that the static entry point's scratch holds (as its declaration states the sizes)."""
    row = (8 * (N + W + 3 * D) + 4 * D * (M + 3) + 16 + 127) // 128 * 128 + 128
    return max(1, (STATIC_BYTES - 1024 - 3 * (4 * N + 256)) // row)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _session(w, n, rng):
    """Nodes of one session as (role, predecessors); the family goes by w."""
    if n < 4:
        return [("chain", [i - 1] if i else []) for i in range(n)]
    if w % 3 == 0:  # planner, then coder / tester repairs, then a reviewer chain
        roles = ["planner"] + ["coder", "tester"] * ((n - 2) // 2) + ["reviewer"] * n
        return [(roles[i], [i - 1] if i else []) for i in range(n)]
    if w % 3 == 1:  # planner, parallel researchers, a synthesizer, reviewers
        k = min(8, n - 3) if n <= 11 else 8 + (n - 11) // 2
        nodes = [("planner", [])] + [("researcher", [0])] * k + [("synthesizer", list(range(1, k + 1)))]
        return nodes + [("reviewer", [i - 1]) for i in range(k + 2, n)]
    nodes, prev = [("layer", [])], [0]
    while len(nodes) < n:
        cur = []
        for _ in range(min(int(rng.integers(1, 5)), n - len(nodes))):
            preds = rng.permutation(prev)[:int(rng.integers(1, 3))]
            cur.append(len(nodes))
            nodes.append(("layer", sorted(int(p) for p in preds)))
        prev = cur
    return nodes


def _problem(case, seed):
    rng = np.random.default_rng(seed)
    N, D, M, W = case["N"], case["D"], case["M"], case["W"]
    classes = [CLASSES[(4 * d + 3) // D if D < 4 else 4 * d // D] for d in range(D)]
    cap = np.array([c[0] * GIB for c in classes], np.int64)
    speed, bw = np.array([c[1] for c in classes]), np.array([c[2] for c in classes], np.int64)
    weight = np.array([g * GIB for g in WEIGHTS[:M]], np.int64)
    fit = np.nonzero(weight + 4096 + case["margin"] <= cap.max())[0]
    preds, model, session = [], [], []
    for w in range(W):
        base, roles = len(model), {}
        for role, ps in _session(w, N // W + (w < N % W), rng):
            key = role if role != "layer" else len(model)
            if role == "layer" and ps and rng.random() < 0.5:
                m = model[base + ps[0]]
            else:
                m = roles.setdefault(key, int(rng.choice(fit)))
            preds.append([base + p for p in ps])
            model.append(m)
            session.append(w)
    model = np.array(model)
    lat = np.rint(rng.lognormal(math.log(2e6), 0.8, N)[:, None] * speed).clip(1, 2**31 - 1)
    peak = np.repeat((weight[model] + rng.integers(256, 4097, N))[:, None], D, 1)
    gaps = rng.exponential(case["gap_ms"] * 1e3, W)
    gaps[0] = 0
    prob = SimpleNamespace(
        N=N, D=D, M=M, W=W, pred_off=np.cumsum([0] + [len(p) for p in preds]), pred_idx=np.array([u for p in preds for u in p], np.int64),
        model=model, session=np.array(session), arrival_us=np.rint(np.cumsum(gaps)).astype(np.int64), lat_us=lat.reshape(-1),
        peak_mib=peak.reshape(-1), weight_mib=weight, load_us=(weight[:, None] * (1 << 20)) // (bw * 1000), cap_mib=cap,
        grant_us=case["grant"], S=case["S"], seed=seed, margin_mib=case["margin"], reclaim=int(case["kind"] == "next_use"),
        batch=case["B"])
    if case["S"]:  # integer Box-Muller tables: radius, angle, exp(0.3 z)
        i = np.arange(4096)
        r = np.rint(4096 * np.sqrt(-2 * np.log((i + 0.5) / 4096))).astype(np.int64)
        c = np.rint(16384 * np.cos(2 * np.pi * i / 4096)).astype(np.int64)
        z = -((-int(r.max()) * 16384) >> 18)
        prob.bm_r, prob.bm_c, prob.bm_e = r, c, np.rint(65536 * np.exp(0.3 * (np.arange(2 * z + 1) - z) / 256)).astype(np.int64)
    return prob, preds


def _pack(bits):
    """bool [P, 32 * words] to int32 [P, words]."""
    w = bits.view(bits.shape[0], -1, 32).to(torch.int64) << torch.arange(32, device=bits.device)
    return w.sum(2).to(torch.int32)  # wraps to the same 32 bits


def _plans(case, prob, preds, gen):
    """P plans on the GPU: a position's sort key is the largest random number among the node and its ancestors, and ties keep the
    node order, which is topological; that is the order in which a scheduler with random priorities takes ready nodes."""
    N, P = case["N"], case["P"]
    plans = wf.DevicePlans.empty(P, N, with_retain=case["retain"])
    fits = torch.from_numpy((prob.peak_mib.reshape(N, -1) + case["margin"] <= prob.cap_mib)).to(DEV)
    count = fits.sum(1)
    devs = torch.argsort(fits.to(torch.int8), dim=1, descending=True, stable=True).to(torch.uint8)  # the fitting devices first
    level = np.zeros(N, np.int64)
    for v in range(N):
        level[v] = 1 + max((level[u] for u in preds[v]), default=-1)
    rounds = []  # (nodes, their j-th predecessors), level by level
    for lv in range(1, int(level.max()) + 1):
        nodes = np.nonzero(level == lv)[0]
        for j in range(max(len(preds[v]) for v in nodes)):
            at = [v for v in nodes if len(preds[v]) > j]
            rounds.append((torch.tensor(at, device=DEV), torch.tensor([preds[v][j] for v in at], device=DEV)))
    low = N.bit_length()
    node = torch.arange(N, device=DEV, dtype=torch.int32)[:, None]
    step = max(1, min(P, (1 << 25) // N))
    for lo in range(0, P, step):
        hi = min(P, lo + step)
        key = torch.randint(0, 1 << (31 - low), (N, hi - lo), device=DEV, dtype=torch.int32, generator=gen)
        for v, u in rounds:
            key[v] = torch.maximum(key[v], key[u])
        key = torch.sort(((key << low) | node).t().contiguous(), dim=1).values
        plans.order[lo:hi].zero_()
        plans.order[lo:hi, :N] = (key & ((1 << low) - 1)).to(torch.int16)
        pick = torch.rand((hi - lo, N), device=DEV, generator=gen)
        pick = torch.minimum((pick * count).long(), count - 1)
        plans.place[lo:hi].zero_()
        plans.place[lo:hi, :N] = devs[torch.arange(N, device=DEV), pick]
        for rows, p in ((plans.fuse, 0.5), (plans.prefetch, 0.5), (plans.retain, 0.8)):
            if rows is not None:
                bits = torch.rand((hi - lo, rows.shape[1] * 32), device=DEV, generator=gen) < p
                bits[:, N:] = False
                rows[lo:hi] = _pack(bits)
    if case["bad"]:  # plans that name a device which is not there
        n = max(1, int(P * case["bad"]))
        plans.place[torch.randperm(P, device=DEV, generator=gen)[:n], N // 2] = 200
    return plans


def _host(t):
    return None if t is None else t.cpu().pin_memory()


def prepare(case, seed):
    prob, preds = _problem(case, seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    kind, P, N, k = case["kind"], case["P"], case["N"], case["k"]
    st = SimpleNamespace(kind=kind, P=P, k=k, seed=seed, jitter=case["jitter"], n_ops=case["n_ops"], round=0)
    def i64(*shape):
        return torch.empty(shape, dtype=torch.int64, device=DEV)

    st.ids, st.keys = torch.empty(k, dtype=torch.int32, device=DEV), i64(k, 3)
    if kind == "static":
        st.prob = wf.DeviceProblem(prob)
        st.plans, st.res = _plans(case, prob, preds, gen), wf.Results(P)
        return st
    st.ctx = wf.Ctx(prob, max_P=P + k)
    if kind == "construct":
        st.plans = wf.DevicePlans.empty(P, N, with_retain=case["retain"])
        for t in (st.plans.place, st.plans.order, st.plans.fuse, st.plans.prefetch, st.plans.retain):
            if t is not None:
                t.zero_()  # the padding, which the call does not write
        return st
    st.plans, st.res = _plans(case, prob, preds, gen), wf.Results(P)
    st.rel, st.comp = i64(N), i64(N)
    if kind == "host":
        p = st.plans
        st.plans = wf.DevicePlans(*(_host(t) for t in (p.place, p.order, p.fuse, p.prefetch, p.retain)))
        st.res = wf.Results(P, device="cpu")
        st.ids, st.keys, st.rel, st.comp = (_host(t) for t in (st.ids, st.keys, st.rel, st.comp))
        wf.wf_ctx_reserve_host(st.ctx)
    elif kind == "phi":
        st.timely, st.life = i64(P), i64(P)
    elif kind == "search":  # the elite: the k best of the batch, whose rows then take the children
        p = st.plans
        wf.wf_eval_plans(st.ctx, p, st.res)
        wf.wf_topk(st.ctx, st.res, P, k, st.ids, st.keys)
        at = st.ids.long()
        st.elite = wf.DevicePlans(*(None if t is None else t[at].contiguous() for t in (p.place, p.order, p.fuse, p.prefetch, p.retain)))
        st.elite_res = wf.Results(k)
        for name in ("makespan", "p95", "gpu", "status"):
            getattr(st.elite_res, name).copy_(getattr(st.res, name)[at])
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def _metrics(res):
    return {"makespan": res.makespan, "p95": res.p95, "gpu": res.gpu, "status": res.status}


def _rows(p):
    return {"place": p.place, "order": p.order, "fuse": p.fuse, "prefetch": p.prefetch, "retain": p.retain}


def run(st):
    top = {"ids": st.ids, "keys": st.keys}
    if st.kind == "static":
        wf.wf_eval_plans_static(st.prob, st.plans, st.res)
        return _metrics(st.res)
    if st.kind == "construct":
        wf.wf_construct_plans(st.ctx, st.plans, st.seed, st.jitter)
        return _rows(st.plans)
    if st.kind == "search":  # the next round of a search in progress
        wf.wf_local_search(st.ctx, st.elite, st.elite_res, st.plans, st.res, st.seed, st.round, 1, st.n_ops)
        st.round += 1
        return {"elite": _rows(st.elite), "elite_results": _metrics(st.elite_res), "results": _metrics(st.res)}
    forecast = {"rel": st.rel, "comp": st.comp}
    if st.kind == "host":
        wf.wf_eval_topk_host(st.ctx, st.plans, st.k, st.ids, st.keys, st.res, st.rel, st.comp)
        return {**_metrics(st.res), **top, **forecast}
    if st.kind == "phi":
        wf.wf_eval_plans_phi(st.ctx, st.plans, st.res, st.timely, st.life)
        wf.wf_topk_phi(st.ctx, st.res, st.timely, st.life, st.P, st.k, st.ids, st.keys)
        return {**_metrics(st.res), **top, "timely": st.timely, "life": st.life}
    if st.kind == "step":
        wf.wf_forecast_readiness(st.ctx, st.rel, st.comp)
    wf.wf_eval_plans(st.ctx, st.plans, st.res)
    wf.wf_topk(st.ctx, st.res, st.P, st.k, st.ids, st.keys)
    return {**_metrics(st.res), **top, **(forecast if st.kind == "step" else {})}


def work(case):
    """Bytes: every plan row read (or written) once, the window's tables read once, every result written once.  Operations, all on
    integers: per plan-position about 55 (unit record 15, residency 20, times 20); with samples the times and a hash of 30 for each;
    the constructor scores every device of a position and hashes a jitter for it."""
    N, D, M, W, P, k, S = (case[x] for x in ("N", "D", "M", "W", "P", "k", "S"))
    row = 3 * N + (3 if case["retain"] else 2) * ((N + 7) // 8)
    tables = N * (8 * D + 16) + 4 * M * D + 8 * W
    out = 28 * P + 28 * k + (16 * N if case["kind"] in ("step", "host") else 16 * P if case["kind"] == "phi" else 0)
    ops = N * P * (35 + (50 * S if S else 20))
    if case["kind"] == "construct":
        out, ops = 0, N * P * (40 + D * (60 if case["jitter"] else 10))
    if case["kind"] == "search":
        out += row * P  # the children, written and read
    return {"bytes": row * P + tables + out, "flops": ops}


def tolerance(case):
    return "exact"


# ---------------------------------------------------------------------------
# The same results in plain torch, 64-bit integers, one dispatch position of all plans at a time
# ---------------------------------------------------------------------------

def exact(case, seed):
    """What run() returns, for the evaluations under least-recently-used reclamation with at most 3,000 activations; None for the
    others: reclamation by next use, the replica batch limit, construction and search decide by whole numbers throughout, and their
    results are compared bit for bit."""
    if case["kind"] not in ("step", "host", "phi", "stochastic", "static") or case["N"] > 3000 or case["P"] * max(1, case["S"]) > 1 << 20:
        return None
    prob, preds = _problem(case, seed)
    plans = _plans(case, prob, preds, torch.Generator(device=DEV).manual_seed(seed))
    play = _play(case, prob, preds, plans)
    bad = (plans.place[:, :case["N"]] >= case["D"]).any(1)
    big = torch.iinfo(torch.int64).max
    play = {name: torch.where(bad, big, v) for name, v in play.items()}
    out = {**{n: play[n] for n in ("makespan", "p95", "gpu")}, "status": bad.to(torch.int32)}
    if case["kind"] == "static":
        return out
    if case["kind"] == "phi":
        out.update(timely=play["timely"], life=play["life"])
        terms, key = (play["makespan"], -play["timely"], play["life"]), ("makespan", "timely", "life")
    else:
        terms, key = (play["makespan"], play["p95"], play["gpu"]), ("makespan", "p95", "gpu")
    ids = np.lexsort([t.cpu().numpy() for t in (*terms[::-1], bad.to(torch.int8))])[:case["k"]]
    at = torch.from_numpy(ids.copy()).to(DEV)
    out.update(ids=at.to(torch.int32), keys=torch.stack([play[n][at] for n in key], 1))
    if case["kind"] in ("step", "host"):
        fast = np.where(prob.peak_mib.reshape(case["N"], -1) + case["margin"] <= prob.cap_mib, prob.lat_us.reshape(case["N"], -1), np.inf).min(1)
        rel, comp = np.zeros(case["N"], np.int64), np.zeros(case["N"], np.int64)
        for v in range(case["N"]):
            rel[v] = max([prob.arrival_us[prob.session[v]]] + [comp[u] for u in preds[v]])
            comp[v] = rel[v] + int(fast[v])
        out.update(rel=torch.from_numpy(rel), comp=torch.from_numpy(comp))
    return out


def _i64(x):
    """A Python whole number as the 64-bit pattern that torch takes."""
    return x - (1 << 64) if x >> 63 else x


def _mix(x):
    """The output function of SplitMix64 (Steele, Lea and Flood 2014) on int64 tensors."""
    def shr(v, n):
        return (v >> n) & ((1 << (64 - n)) - 1)
    x = x + _i64(0x9E3779B97F4A7C15)
    x = (x ^ shr(x, 30)) * _i64(0xBF58476D1CE4E5B9)
    x = (x ^ shr(x, 27)) * _i64(0x94D049BB133111EB)
    return x ^ shr(x, 31)


def _play(case, prob, preds, plans):
    N, D, M, W, P, S = (case[x] for x in ("N", "D", "M", "W", "P", "S"))

    def dev(x):
        return torch.as_tensor(np.asarray(x).astype(np.int64), device=DEV)
    place = plans.place[:, :N].long().clamp(max=D - 1)  # (plans that name no device are marked by the caller)
    order = plans.order[:, :N].long() & 0xFFFF
    words = torch.arange(N, device=DEV)

    def unpack(rows):
        return ((rows.long()[:, words >> 5] >> (words & 31)) & 1).bool()
    fuse, prefetch = unpack(plans.fuse), unpack(plans.prefetch)
    retain = unpack(plans.retain) if plans.retain is not None else None
    succ = [[] for _ in range(N)]
    for v in range(N):
        for u in preds[v]:
            succ[u].append(v)
    fnext = [succ[u][0] if len(succ[u]) == 1 and preds[succ[u][0]] == [u] and prob.model[u] == prob.model[succ[u][0]] else -1 for u in range(N)]
    fprev = np.full(N, -1)
    for u, v in enumerate(fnext):
        if v >= 0:
            fprev[v] = u
    fnext, fprev = dev(fnext), dev(fprev)
    most = max(1, max(len(p) for p in preds))
    pred = dev([p + [N] * (most - len(p)) for p in preds])  # N: a finish of 0
    model, session, arrival = dev(prob.model), dev(prob.session), dev(prob.arrival_us)
    lat, kv_of = dev(prob.lat_us).view(N, D), dev(prob.peak_mib + case["margin"]).view(N, D) - dev(prob.weight_mib)[model][:, None]
    weight, load, cap = dev(prob.weight_mib), dev(prob.load_us).view(M, D), dev(prob.cap_mib)
    rows = torch.arange(P, device=DEV)
    L = max(1, S)
    if S:
        key = _mix(_mix(_i64(int(prob.seed)) ^ rows)[:, None] ^ torch.arange(S, device=DEV))
        bm_r, bm_c, bm_e = dev(prob.bm_r), dev(prob.bm_c), dev(prob.bm_e)

    def run_of(v, d):
        base = lat[v, d][:, None]
        if not S:
            return base
        h = _mix(key ^ v[:, None])
        z = (bm_r[h & 4095] * bm_c[(h >> 32) & 4095]) >> 18
        return (base * bm_e[z + (len(prob.bm_e) - 1) // 2] + 32768) >> 16

    def zeros(*s):
        return torch.zeros(s, dtype=torch.int64, device=DEV)
    finish, tfree, comp = zeros(P, N + 1, L), zeros(P, D, L), zeros(P, W, L)
    stamp, used, ever = zeros(P, D, M), zeros(P, D), torch.zeros((P, D, M), dtype=torch.bool, device=DEV)
    nres, opened, gpu, timely, life = zeros(P, D), zeros(P, D, L), zeros(P, L), zeros(P), zeros(P)
    for i in range(N):
        h = order[:, i]
        d = place[rows, h]
        fp = fprev[h]
        unit = ~((fp >= 0) & fuse[rows, h] & (place[rows, fp.clamp(min=0)] == d))
        m, arr = model[h], arrival[session[h]][:, None]
        rel = torch.maximum(arr, finish[rows[:, None], pred[h]].amax(1))
        run, kv, tail, s = run_of(h, d), kv_of[h, d], h, fnext[h]
        while True:
            c = s.clamp(min=0)
            on = unit & (s >= 0) & fuse[rows, c] & (place[rows, c] == d)
            if not bool(on.any()):
                break
            run = torch.where(on[:, None], run + run_of(c, d), run)
            kv = torch.where(on, torch.maximum(kv, kv_of[c, d]), kv)
            tail, s = torch.where(on, c, tail), torch.where(on, fnext[c], torch.full_like(s, -1))
        hit = stamp[rows, d, m] > 0
        need = kv + torch.where(hit, 0, weight[m])
        empty = nres[rows, d] == 0
        while True:  # the least recently used other model leaves
            over = unit & (used[rows, d] + need > cap[d])
            if not bool(over.any()):
                break
            age = torch.where(stamp[rows, d] > 0, stamp[rows, d], N + 9).scatter(1, m[:, None], N + 9)
            v = age.argmin(1)
            stamp[rows, d, v] = torch.where(over, 0, stamp[rows, d, v])
            used[rows, d] -= torch.where(over, weight[v], 0)
            nres[rows, d] -= over.long()
        tf, pf = tfree[rows, d], prefetch[rows, h]
        ls = torch.maximum(tf, torch.where(pf[:, None], arr, rel))
        le = ls + load[m, d][:, None]
        ready = torch.maximum(tf, rel)
        start = torch.where(hit[:, None], ready, torch.maximum(le, rel))
        miss = unit & ~hit
        timely += (miss & pf & (ls < rel)[:, 0] & (le <= rel)[:, 0]).long()
        life += torch.where(unit, (start - ready)[:, 0] + torch.where(miss & ever[rows, d, m], load[m, d], 0), 0)
        ever[rows, d, m] |= miss
        first = miss & empty
        opened[rows, d] = torch.where(first[:, None], ls, opened[rows, d])
        used[rows, d] += torch.where(miss, weight[m], 0)
        nres[rows, d] += miss.long()
        end = start + case["grant"] + run
        at = torch.where(unit, tail, N)
        finish[rows, at] = torch.where(unit[:, None], end, 0)
        tfree[rows, d] = torch.where(unit[:, None], end, tf)
        w = session[h]
        comp[rows, w] = torch.where(unit[:, None], torch.maximum(comp[rows, w], end), comp[rows, w])
        gone = unit & ~retain[rows, tail] if retain is not None else torch.zeros_like(unit)
        stamp[rows, d, m] = torch.where(unit, torch.where(gone, 0, i + 1), stamp[rows, d, m])
        used[rows, d] -= torch.where(gone, weight[m], 0)
        nres[rows, d] -= gone.long()
        gpu += torch.where((gone & (nres[rows, d] == 0))[:, None], end - opened[rows, d], 0)
    last = comp.amax(1)
    gpu += torch.where((nres > 0)[:, :, None], last[:, None] - opened, 0).sum(1)
    pool = (comp - arrival[None, :, None]).reshape(P, -1).sort(1).values
    return {"makespan": (last - arrival.min()).sum(1) // L, "p95": pool[:, (95 * W * L + 99) // 100 - 1], "gpu": gpu.sum(1) // L,
            "timely": timely, "life": life}
