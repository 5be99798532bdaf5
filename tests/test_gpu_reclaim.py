"""Bit-exact parity of reclamation by next use with the oracle."""
import numpy as np
import pytest

import oracle
import wfgen
from gpu_util import assert_same, gpu_eval, lib, oracle_eval
from randprob import random_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,P", [("tiny", 1024), ("mix", 4096), ("burst", 2048)])
def test_named_workloads(name, P):
    w = wfgen.config(name)
    prob = w.problem.with_(reclaim=1)
    plans = wfgen.make_plans(prob, P, w.plan_seed)
    got = gpu_eval(prob, plans, k=16)
    want = oracle_eval(prob, plans)
    assert_same(got, want)
    lru = oracle_eval(w.problem, plans)
    assert not np.array_equal(want["makespan"], lru["makespan"]) or name == "tiny"


@pytest.mark.parametrize("seed", range(6))
def test_random_windows(seed):
    rng = np.random.default_rng(3100 + seed)
    prob = random_problem(rng, n_sessions=int(rng.integers(1, 7)), D=int(rng.integers(1, 6)),
                          M=int(rng.integers(2, 16 if seed == 5 else 8))).with_(reclaim=1)
    if seed % 2:
        prob = prob.with_(grant_us=int(rng.integers(1, 300)))
    plans = wfgen.make_plans(prob, int(rng.integers(1, 400)), seed, p_retain=0.5 if seed % 3 else None)
    from test_gpu_parity import inject_invalid
    if plans.P >= 8:
        inject_invalid(plans, prob, rng)
    assert_same(gpu_eval(prob, plans), oracle_eval(prob, plans))


def test_overflowing_times_keep_the_policy():
    """Times beyond 2^32 us move plans to the 64-bit sweep, which applies the
    same reclamation order."""
    rng = np.random.default_rng(53)
    prob = random_problem(rng, n_sessions=5, sizes=(6, 10), D=2, M=4)
    lat = prob.lat_us.astype(np.int64).reshape(prob.N, prob.D)
    lat[:2, 1] = (1 << 31) - 1
    prob = prob.with_(lat_us=lat.astype(np.int32).reshape(-1), reclaim=1)
    plans = wfgen.make_plans(prob, 300, 7)
    want = oracle_eval(prob, plans)
    mk = want["makespan"][want["status"] == 0]
    assert (mk >= (1 << 32)).any() and (mk < (1 << 31)).any()
    assert_same(gpu_eval(prob, plans), want)


def test_policy_switch_on_one_context():
    import torch
    wf = lib()
    w = wfgen.config("mix")
    plans = wfgen.make_plans(w.problem, 512, 3)
    ctx = wf.Ctx(w.problem, max_P=512)
    dp = wf.DevicePlans.from_host(plans, "cuda")
    outs = []
    for pol in (0, 1, 0, 1):
        wf.wf_ctx_set_reclaim(ctx, pol)
        res = wf.Results(512)
        wf.wf_eval_plans(ctx, dp, res)
        torch.cuda.synchronize()
        outs.append(res.numpy())
    for a, b in zip(outs[0], outs[2]):
        assert np.array_equal(a, b)
    for a, b in zip(outs[1], outs[3]):
        assert np.array_equal(a, b)
    want = oracle.eval_plans(w.problem.with_(reclaim=1), plans, threads=8)
    assert np.array_equal(outs[1][0], want[0]) and np.array_equal(outs[1][2], want[2])


def test_stochastic_problems_refuse_the_policy():
    wf = lib()
    w = wfgen.config("stochastic")
    ctx = wf.Ctx(w.problem, max_P=8)
    with pytest.raises(wf.WfError):
        wf.wf_ctx_set_reclaim(ctx, 1)


@pytest.mark.parametrize("loads", ["zero", "equal", "powers", "near", "huge"])
@pytest.mark.parametrize("D,M", [(3, 7), (6, 8), (32, 9), (5, 16)])
def test_tied_and_nearly_tied_quotients(loads, D, M):
    """Reload costs whose quotients tie exactly (all equal, powers of two), come
    within a few units in the last place of a float (2^24 + a little, and up
    to 2^31 - 1), or are infinite (no reload cost)."""
    rng = np.random.default_rng(3200 + 10 * D + M)
    prob = random_problem(rng, n_sessions=9, sizes=(8, 16), D=D, M=M)
    m = np.arange(M)[:, None] + np.zeros((1, D), np.int64)
    load = {"zero": m * 0, "equal": m * 0 + 48, "powers": 1 << (m % 6), "near": (1 << 24) * (1 + m % 3) + rng.integers(0, 3, (M, D)),
            "huge": (1 << 31) - 1 - rng.integers(0, 4, (M, D)) * (1 + m % 2)}[loads]
    prob = prob.with_(reclaim=1, load_us=load.reshape(-1).astype(np.int32))
    plans = wfgen.make_plans(prob, 200, D + M, p_retain=0.7 if D % 2 else None)
    assert_same(gpu_eval(prob, plans), oracle_eval(prob, plans))


@pytest.mark.parametrize("D,M,P,scale", [(1, 1, 5, 1), (4, 2, 333, 1), (3, 3, 200, 1), (9, 4, 100, 1), (32, 4, 33, 1), (3, 5, 100, 1),
                                         (2, 4, 100, 400000), (4, 1, 100, 1 << 20)])
def test_few_models(D, M, P, scale):
    """Four lanes a plan up to four models (and five models on eight lanes),
    with retain rows, invalid plans and run times that leave 32 bits."""
    rng = np.random.default_rng(3400 + 10 * D + M)
    prob = random_problem(rng, n_sessions=12, sizes=(6, 12), D=D, M=M)
    prob = prob.with_(reclaim=1, lat_us=np.minimum(prob.lat_us.astype(np.int64) * scale, (1 << 28)).astype(np.int32))
    plans = wfgen.make_plans(prob, P, M, p_retain=0.7 if D % 2 else None)
    if P > 8:
        plans.place[3, 1] = D
        plans.order[5, 0] = plans.order[5, 1]
    assert_same(gpu_eval(prob, plans), oracle_eval(prob, plans))


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 96, 97])
def test_window_lengths_of_the_next_use_pass(n):
    """One to four chunks of 32 positions: the pass without reads ahead (up to
    64 activations) and with them, chains that fuse across chunks."""
    from test_gpu_edges import chains_window
    prob = chains_window([n - n // 2, n // 2] if n > 1 else [1], D=2, M=1, seed=n)
    rng = np.random.default_rng(n)
    prob = prob.with_(reclaim=1, M=3, model=np.sort(rng.integers(0, 3, n)).astype(np.uint8), weight_mib=np.array([2, 3, 4], np.int32),
                      peak_mib=np.full(2 * n, 6, np.int32), load_us=rng.integers(1, 100, 6).astype(np.int32))
    plans = wfgen.make_plans(prob, 150, n)
    assert_same(gpu_eval(prob, plans), oracle_eval(prob, plans))


@pytest.mark.parametrize("D,M,scale,shift", [(2, 5, 1, 0), (8, 8, 1, 0), (9, 9, 1, 0), (32, 16, 1, 0), (4, 6, 400000, 3_000_000_000),
                                             (3, 12, 1 << 20, 1_500_000_000)])
def test_short_windows_in_large_batches(D, M, scale, shift):
    """Batches of more than 40 plans an SM, where windows up to a length take a
    lane per plan: the longest such window and the next longer one, the batch at
    the limit and one plan more; all rules of the order, window terms, retain
    rows, invalid plans, run times that leave 32 bits."""
    import torch
    from test_gpu_phi import check
    most = 40 * torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(3500 + 10 * D + M)
    limit = 24 + 2 * D if M <= 8 else 32 + 8 * D
    for n in (limit, limit + 1, 9):
        cuts = [n] if n < 20 else [n // 3, n // 3, n - 2 * (n // 3)]
        sess = [(wfgen.fam_softdev(c), wfgen.fam_research(c, width=3), wfgen.fam_layered(c, rng, width=3))[i % 3] for i, c in enumerate(cuts)]
        dev = wfgen.DeviceSpec(cap_gib=[(60 + 7 * d) / wfgen.GIB for d in range(D)], speed=[1.0 + 0.1 * d for d in range(D)], bw_gbps=[1] * D)
        prob = wfgen.assemble("short", sess, shift + np.sort(rng.integers(0, 300, len(sess))).astype(np.int64), dev,
                              [(5 + (7 * m) % 31) / wfgen.GIB for m in range(M)], rng, lat_median_us=100, lat_sigma=0.6, kv_lo=1, kv_hi=20)
        assert prob.N == n
        prob = prob.with_(load_us=rng.integers(0, 60, M * D).astype(np.int32), reclaim=1,
                          lat_us=np.minimum(prob.lat_us.astype(np.int64) * scale, 1 << 26).astype(np.int32))
        plans = wfgen.make_plans(prob, most + 1, D + M, p_retain=0.8 if D % 2 else None)
        plans.place[7, 0] = D
        plans.order[11, 0] = plans.order[11, 1]
        got = check(prob, plans, k=8, reclaim=1)
        plain = gpu_eval(prob, plans)
        assert_same(plain, got)
        assert_same(gpu_eval(prob, plans.slice(0, most)), {x: got[x][:most] for x in ("status", "makespan", "p95", "gpu")})


@pytest.mark.parametrize("n,sessions", [(96, 3), (97, 3), (96, 1), (95, 3), (64, 2)])
def test_long_sessions_in_large_batches(n, sessions):
    """Up to eight models, windows of up to 96 activations take a lane per plan
    when their sessions have 32 or more: at and around both limits."""
    import torch
    P = 40 * torch.cuda.get_device_properties(0).multi_processor_count + 1
    rng = np.random.default_rng(3600 + n + sessions)
    prob = random_problem(rng, n_sessions=sessions, sizes=(n // sessions,) * 2, D=3, M=6)
    while prob.N != n:  # (the families round some sizes)
        prob = random_problem(rng, n_sessions=sessions, sizes=(n // sessions, n // sessions + (n % sessions > 0)), D=3, M=6)
    prob = prob.with_(reclaim=1)
    plans = wfgen.make_plans(prob, P, n)
    plans.place[7, 0] = 3
    assert_same(gpu_eval(prob, plans), oracle_eval(prob, plans))


@pytest.mark.parametrize("M", [8, 9, 16])
def test_batches_of_one_wave_of_four_ctas(M):
    """Beyond eight models, batches between three and four CTAs an SM take a lane
    per plan on longer windows too: both ends of that range and one plan beyond
    each."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(3800 + M)
    prob = random_problem(rng, n_sessions=20, sizes=(6, 12), D=4, M=M).with_(reclaim=1)
    assert prob.N > 32 + 8 * 4
    plans = wfgen.make_plans(prob, 64 * sms + 1, 3, p_retain=0.8)
    want = oracle_eval(prob, plans)
    for P in (48 * sms, 48 * sms + 1, 64 * sms, 64 * sms + 1):
        assert_same(gpu_eval(prob, plans.slice(0, P)), {x: want[x][:P] for x in ("status", "makespan", "p95", "gpu")})


def lone_sessions(W, D, M, seed):
    """W sessions of one activation each: as many finish slots as sessions."""
    rng = np.random.default_rng(seed)
    dev = wfgen.DeviceSpec(cap_gib=[60 + d for d in range(D)], speed=[1.0] * D, bw_gbps=[1] * D)
    prob = wfgen.assemble("wide", [[("planner", [])] for _ in range(W)], np.sort(rng.integers(0, 500, W)).astype(np.int64), dev,
                          [5 + m for m in range(M)], rng, lat_median_us=100, lat_sigma=0.6, kv_lo=1, kv_hi=20)
    prob = prob.with_(model=rng.integers(0, M, W).astype(prob.model.dtype))
    return prob.with_(peak_mib=np.repeat(prob.weight_mib[prob.model] + 64, D).astype(np.int32))


@pytest.mark.parametrize("D,M", [(1, 1), (2, 2), (3, 4), (2, 6), (7, 8), (5, 12), (32, 16)])
def test_last_window_that_takes_the_policy(D, M):
    """The windows that take the policy are those whose state for three plans
    (a queue word and 16-bit next uses per plan and device) fits a CTA's
    227 KiB, whatever the layout of the sweep that plays them: the largest
    one takes it and gives the oracle's results, the next refuses it."""
    wf = lib()
    r16 = lambda x: (x + 15) & ~15
    queue = 12 if M <= 8 else 24

    def size(W):
        return (r16(4 * M) + r16(4 * D) + r16(4 * M * D) + r16(4 * W) + 4608 + r16(24 * (W + 2)) + r16(24 * D) + r16(queue * D) +
                r16(12 * D) + r16(3 * D) + 32 + r16(6 * D * M) + r16(3 * M) + 48)
    W = next(w for w in range(9000, 1, -1) if size(w) <= 227 * 1024)
    prob = lone_sessions(W, D, M, 10 * D + M)
    plans = wfgen.make_plans(prob, 4, 1)
    assert_same(gpu_eval(prob.with_(reclaim=1), plans), oracle_eval(prob.with_(reclaim=1), plans))
    ctx = wf.Ctx(lone_sessions(W + 1, D, M, 10 * D + M), max_P=4)
    with pytest.raises(wf.WfError) as e:
        wf.wf_ctx_set_reclaim(ctx, 1)
    assert e.value.code == wf.WF_EINVAL
    ctx.close()


def test_largest_window():
    """A window near the shared-memory limit of the policy (32 devices, 16
    models, 7,800 sessions), where the sweep plays two plans per CTA."""
    rng = np.random.default_rng(3300)
    W, D, M = 7800, 32, 16
    dev = wfgen.DeviceSpec(cap_gib=[60 + d for d in range(D)], speed=[1.0] * D, bw_gbps=[1] * D)
    prob = wfgen.assemble("wide", [[("planner", [])] for _ in range(W)], np.sort(rng.integers(0, 500, W)).astype(np.int64), dev,
                          [5 + m for m in range(M)], rng, lat_median_us=100, lat_sigma=0.6, kv_lo=1, kv_hi=20)
    prob = prob.with_(reclaim=1, model=rng.integers(0, M, W).astype(prob.model.dtype))
    prob = prob.with_(peak_mib=np.repeat(prob.weight_mib[prob.model] + 64, D).astype(np.int32))
    plans = wfgen.make_plans(prob, 5, 1)
    assert_same(gpu_eval(prob, plans), oracle_eval(prob, plans))
