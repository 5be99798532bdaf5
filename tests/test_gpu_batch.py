"""GPU parity for the replica batch limit B_q (wf_ctx_set_batch): the replica
batch sweep and the int64 path's batched play against the oracle's, element by
element."""
import numpy as np
import pytest

import oracle
import wfgen
from golden_util import fixture_names, load, plans_of, problem_of
from gpu_util import THREADS, assert_same, gpu_eval, lib, oracle_eval
from randprob import random_problem
from test_gpu_parity import inject_invalid

pytestmark = pytest.mark.gpu


def _gpu(prob, plans, k=None):
    wf = lib()
    ctx = wf.Ctx(prob, max_P=plans.P)  # the context takes prob.batch (wf_ctx_set_batch)
    out = gpu_eval(prob, plans, k=k, ctx=ctx)
    ctx.close()
    return out


@pytest.mark.parametrize("seed", range(8))
def test_random_windows(seed):
    rng = np.random.default_rng(3100 + seed)
    B = [1, 2, 3, 5][seed % 4]
    prob = random_problem(rng, n_sessions=int(rng.integers(2, 7)), D=int(rng.integers(1, 5)),
                          M=int(rng.integers(1, 6)), tight=bool(seed % 2)).with_(batch=B)
    plans = wfgen.make_plans(prob, int(rng.integers(50, 400)), seed, p_retain=0.6 if B == 1 else None)
    inject_invalid(plans, prob, rng)
    got = _gpu(prob, plans, k=8)
    want = oracle_eval(prob, plans)
    assert_same(got, want)
    ids, keys = oracle.topk(want["makespan"], want["p95"], want["gpu"], want["status"], 8)
    assert np.array_equal(got["ids"], ids) and np.array_equal(got["keys"], keys)


@pytest.mark.parametrize("name", [n for n in fixture_names() if n.startswith(("t10", "t11", "t12"))])
def test_hand_worked_windows(name):
    fx = load(name)
    for case in fx["cases"]:
        prob = problem_of(fx, case)
        plans = plans_of(fx, [case])
        got = _gpu(prob, plans)
        exp = case["expect"]
        assert (int(got["makespan"][0]), int(got["p95"][0]), int(got["gpu"][0])) == \
            (exp["makespan"], exp["p95"], exp["gpu"]), case["label"]


@pytest.mark.parametrize("B", [1, 2, 4])
def test_burst_window_in_full(B):
    w = wfgen.config("burst")
    prob = w.problem.with_(batch=B)
    plans = wfgen.make_plans(prob, w.P, w.plan_seed)
    got = _gpu(prob, plans, k=w.k)
    want = oracle_eval(prob, plans)
    assert_same(got, want)


def test_batch_one_equals_the_sweep():
    """B_q = 1 gives the results of the sweep without a limit."""
    w = wfgen.config("mix")
    plans = wfgen.make_plans(w.problem, 8192, 4)
    a = gpu_eval(w.problem, plans)
    b = _gpu(w.problem.with_(batch=1), plans)
    assert_same(b, a)


@pytest.mark.parametrize("D,M,B,P", [(1, 1, 1, 1), (8, 8, 4, 65), (8, 9, 5, 7), (9, 8, 4, 33), (16, 16, 64, 9),
                                     (17, 8, 3, 8), (32, 16, 5, 17)])
def test_lanes_per_plan(D, M, B, P):
    """8, 16 and 32 lanes per plan, both queue words, running slots in
    registers and in shared memory, CTAs whose plans are not all there."""
    rng = np.random.default_rng(10 * D + B)
    prob = random_problem(rng, n_sessions=40, D=D, M=M).with_(batch=B)
    plans = wfgen.make_plans(prob, P, 3, p_retain=0.6 if B == 1 else None)
    assert_same(_gpu(prob, plans), oracle_eval(prob, plans))


@pytest.mark.parametrize("D,M,B,P", [(17, 3, 1, 40), (17, 9, 4, 1000), (24, 8, 5, 333), (31, 16, 4, 64), (32, 8, 64, 9), (32, 5, 2, 2000)])
def test_two_devices_a_lane(D, M, B, P):
    """Beyond 16 devices a lane plays two of them in turn: windows long enough
    that both are used and exchanged often, running slots in registers and in
    shared memory, retain rows, some invalid plans."""
    rng = np.random.default_rng(D + B)
    prob = random_problem(rng, n_sessions=60, D=D, M=M).with_(batch=B)
    plans = wfgen.make_plans(prob, P, 8, p_retain=0.6 if B == 1 else None)
    inject_invalid(plans, prob, rng)
    assert_same(_gpu(prob, plans), oracle_eval(prob, plans))


@pytest.mark.parametrize("sessions,D,B", [(1, 3, 2), (33, 8, 4), (100, 12, 4), (300, 5, 3), (700, 20, 1)])
def test_p95_over_every_lane_s_sessions(sessions, D, B):
    """A plan's lanes write its sessions' latencies side by side and the whole
    warp then selects among them: fewer sessions than lanes, several a lane,
    more than the selection keeps in registers (256), and a rank beyond its
    taking of maxima (700: the 36th largest)."""
    rng = np.random.default_rng(sessions)
    prob = random_problem(rng, n_sessions=sessions, sizes=(4, 5), D=D, M=4).with_(batch=B)
    plans = wfgen.make_plans(prob, 61, 2)
    assert_same(_gpu(prob, plans), oracle_eval(prob, plans))


@pytest.mark.parametrize("scale,B", [(165000, 2), (1 << 20, 4), (1 << 20, 6), (1 << 24, 1)])
def test_times_past_32_bits(scale, B):
    """Some or all plans leave the 32-bit sweep (and with the largest scale
    some fused chains' run times too): the 64-bit sweep and the int64 path,
    twice on one context (the second call may start on 64-bit times)."""
    wf = lib()
    rng = np.random.default_rng(scale % 97 + B)
    prob = random_problem(rng, n_sessions=30, sizes=(6, 12), D=4, M=5)
    prob = prob.with_(batch=B, lat_us=np.minimum(prob.lat_us.astype(np.int64) * scale, 2**31 - 1).astype(np.int32))
    plans = wfgen.make_plans(prob, 200, 6)
    want = oracle_eval(prob, plans)
    ctx = wf.Ctx(prob, max_P=plans.P)
    for _ in range(2):
        assert_same(gpu_eval(prob, plans, ctx=ctx), want)
    ctx.close()


@pytest.mark.parametrize("D,B", [(3, 4), (12, 6), (24, 2)])
def test_many_plans_past_32_bits(D, B):
    """More plans leave 32 bits than the CTAs of the 64-bit sweep hold at once
    (six an SM of eight plans each), so each walks over several groups; a
    third of the plans stay within 32 bits, and some are invalid."""
    import torch
    P = 60 * torch.cuda.get_device_properties(0).multi_processor_count * 3 // 2
    rng = np.random.default_rng(3700 + D)
    prob = random_problem(rng, n_sessions=2, sizes=(5, 6), D=D, M=5).with_(batch=B)
    base = oracle_eval(prob, wfgen.make_plans(prob, 300, 6))
    ok = base["status"] == 0
    shift = (1 << 32) - int(np.quantile(base["makespan"][ok], 0.3)) - int(prob.arrival_us.min())  # (a third of the plans end below 2^32)
    prob = prob.with_(arrival_us=prob.arrival_us + shift)
    plans = wfgen.make_plans(prob, P, 6)
    inject_invalid(plans, prob, rng, frac=0.02)
    want = oracle_eval(prob, plans)
    end = want["makespan"][want["status"] == 0] + int(prob.arrival_us.min())
    assert 0.1 < (end < (1 << 32)).mean() < 0.6
    assert_same(_gpu(prob, plans), want)


def test_refusals():
    wf = lib()
    import torch
    s = wfgen.config("stochastic").problem
    ctx = wf.Ctx(s, max_P=8)
    with pytest.raises(wf.WfError) as e:
        wf.wf_ctx_set_batch(ctx, 2)
    assert e.value.code == wf.WF_EINVAL
    ctx.close()
    w = wfgen.config("tiny")
    ctx = wf.Ctx(w.problem, max_P=16)
    with pytest.raises(wf.WfError):
        wf.wf_ctx_set_batch(ctx, 65)
    wf.wf_ctx_set_batch(ctx, 2)
    with pytest.raises(wf.WfError):
        wf.wf_ctx_set_reclaim(ctx, 1)
    plans = wfgen.make_plans(w.problem, 16, 1, p_retain=0.5)
    dp = wf.DevicePlans.from_host(plans, "cuda")
    res = wf.Results(16)
    with pytest.raises(wf.WfError) as e:
        wf.wf_eval_plans(ctx, dp, res)
    assert "retain" in str(e.value)
    nr = wf.DevicePlans.from_host(wfgen.make_plans(w.problem, 16, 1), "cuda")
    t = torch.empty(16, dtype=torch.int64, device="cuda")
    with pytest.raises(wf.WfError):
        wf.wf_eval_plans_phi(ctx, nr, res, t, torch.empty_like(t))
    wf.wf_eval_plans(ctx, nr, res)  # the context still works
    wf.wf_ctx_status(ctx)
    ctx.close()
