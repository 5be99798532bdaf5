"""wf_eval_plans_static: the entry point for callers that cannot allocate
device memory (for instance a scheduler inside a serving engine that reserved
almost all GPU memory for weights and KV cache).  Its scratch is the library's
static device array; it must give exactly what the context-based entry point
and the CPU oracle give, call after call, without allocating.  This file is
collected last on purpose."""
import re

import numpy as np
import pytest

import oracle
import wfgen

pytestmark = pytest.mark.gpu


def _both(wf, prob, plans, ctx, dprob):
    import torch
    dp = wf.DevicePlans.from_host(plans, "cuda")
    ref = wf.Results(plans.P)
    wf.wf_eval_plans(ctx, dp, ref)
    got = wf.Results(plans.P)
    wf.wf_eval_plans_static(dprob, dp, got)
    wf.wf_static_status()
    torch.cuda.synchronize()
    return ref.numpy(), got.numpy()


def test_static_entry_matches_context_entry_and_oracle_twice_in_a_row():
    from paper_2609_03335_gb300 import build, wf
    build.build()
    # call 1: the burst window, 1500 plans with some invalid ones
    w1 = wfgen.config("burst")
    p1 = wfgen.make_plans(w1.problem, 1500, 11)
    p1.place[3, 7] = w1.problem.D
    p1.order[9, 0] = p1.order[9, 1]
    ctx1 = wf.Ctx(w1.problem, max_P=p1.P)
    ref1, got1 = _both(wf, w1.problem, p1, ctx1, wf.DeviceProblem(w1.problem))
    # call 2 right after: another window and retain bits
    w2 = wfgen.config("mix")
    p2 = wfgen.make_plans(w2.problem, 5000, 12, p_retain=0.6)
    ctx2 = wf.Ctx(w2.problem, max_P=p2.P)
    ref2, got2 = _both(wf, w2.problem, p2, ctx2, wf.DeviceProblem(w2.problem))
    for ref, got in ((ref1, got1), (ref2, got2)):
        for a, b in zip(ref, got):
            assert np.array_equal(a, b)
    assert got1[3][3] != 0 and got1[3][9] != 0
    # the oracle on a sample of each batch
    for prob, plans, got in ((w1.problem, p1, got1), (w2.problem, p2, got2)):
        sub = plans.slice(0, 300)
        want = oracle.eval_plans(prob, sub)
        for a, b in zip(got, want):
            assert np.array_equal(a[:300], b)
    ctx1.close()
    ctx2.close()


def test_static_entry_allocates_nothing():
    import torch
    from paper_2609_03335_gb300 import build, wf
    build.build()
    w = wfgen.config("mix")
    plans = wfgen.make_plans(w.problem, 2000, 5)
    dprob = wf.DeviceProblem(w.problem)
    dp = wf.DevicePlans.from_host(plans, "cuda")
    out = wf.Results(plans.P)
    wf.wf_eval_plans_static(dprob, dp, out)  # the first call loads the module and looks the array up
    wf.wf_static_status()
    torch.cuda.synchronize()
    free0, _ = torch.cuda.mem_get_info()
    wf.wf_eval_plans_static(dprob, dp, out)
    wf.wf_static_status()
    torch.cuda.synchronize()
    free1, _ = torch.cuda.mem_get_info()
    assert free1 == free0


def test_static_entry_accepts_exactly_the_largest_batch_it_names():
    import torch
    from paper_2609_03335_gb300 import build, wf
    build.build()
    w = wfgen.config("burst")
    plans = wfgen.make_plans(w.problem, 4000, 1)
    dprob = wf.DeviceProblem(w.problem)
    dp = wf.DevicePlans.from_host(plans, "cuda")
    out = wf.Results(plans.P)
    with pytest.raises(wf.WfError) as e:
        wf.wf_eval_plans_static(dprob, dp, out)
    assert e.value.code == wf.WF_EINVAL and "at most" in str(e.value)
    fit = int(re.search(r"at most (\d+) plans", str(e.value)).group(1))
    assert 1000 < fit < plans.P
    wf.wf_eval_plans_static(dprob, wf.DevicePlans.from_host(plans.slice(0, fit), "cuda"), wf.Results(fit))
    wf.wf_static_status()
    torch.cuda.synchronize()
    with pytest.raises(wf.WfError) as e:
        wf.wf_eval_plans_static(dprob, wf.DevicePlans.from_host(plans.slice(0, fit + 1), "cuda"),
                                wf.Results(fit + 1))
    assert e.value.code == wf.WF_EINVAL
    s = wfgen.config("stochastic").problem
    sp = wfgen.make_plans(s, 8, 1)
    with pytest.raises(wf.WfError) as e:
        wf.wf_eval_plans_static(wf.DeviceProblem(s), wf.DevicePlans.from_host(sp, "cuda"), wf.Results(8))
    assert e.value.code == wf.WF_EINVAL


def test_static_entry_reports_tables_that_fail_its_device_check():
    """A model id >= M in the device tables: the device check catches it before
    any table is indexed by it; every plan gets WF_ST_TABLES and INT64_MAX, and
    wf_static_status names the failure.  The next good call is clean."""
    import torch
    from paper_2609_03335_gb300 import build, wf
    build.build()
    w = wfgen.config("tiny")
    plans = wfgen.make_plans(w.problem, 64, 3)
    dp = wf.DevicePlans.from_host(plans, "cuda")
    bad = wf.DeviceProblem(w.problem)
    bad.tensors["model"][5] = w.problem.M  # in bounds of the array; out of the model range
    out = wf.Results(plans.P)
    wf.wf_eval_plans_static(bad, dp, out)
    with pytest.raises(wf.WfError) as e:
        wf.wf_static_status()
    assert e.value.code == wf.WF_EINVAL and "model id" in str(e.value)
    mk, p95, gpu, st = out.numpy()
    assert (st == wf.ST_TABLES).all() and (mk == wf.INT64_MAX).all() and (gpu == wf.INT64_MAX).all()
    good = wf.DeviceProblem(w.problem)
    wf.wf_eval_plans_static(good, dp, out)
    wf.wf_static_status()
    torch.cuda.synchronize()
    want = oracle.eval_plans(w.problem, plans)
    for a, b in zip(out.numpy(), want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("sessions,sizes,D,M,scale", [(1, (4, 4), 1, 1, 1), (8, (4, 4), 3, 8, 1), (11, (3, 3), 32, 9, 1),
                                                      (70, (4, 9), 9, 16, 1), (40, (4, 9), 3, 4, 150000), (3, (5, 9), 2, 3, 1 << 24)])
def test_static_entry_on_edges(sessions, sizes, D, M, scale):
    """Windows of 32 and 33 activations, both queue words, more than 32
    sessions, and run times that leave 32 bits for all or some plans (the
    64-bit replay), against the oracle."""
    from randprob import random_problem
    from paper_2609_03335_gb300 import build, wf
    build.build()
    rng = np.random.default_rng(sessions * 100 + D)
    prob = random_problem(rng, n_sessions=sessions, sizes=sizes, D=D, M=M) if sizes != (3, 3) else \
        random_problem(rng, n_sessions=8, sizes=(4, 4), D=D, M=M)
    if sizes == (3, 3):  # 33 activations
        assert prob.N == 32
        prob = prob.with_(N=33, W=9, pred_off=np.append(prob.pred_off, prob.pred_off[-1]).astype(np.int32),
                          model=np.append(prob.model, 0).astype(np.uint8), session=np.append(prob.session, 8).astype(np.int32),
                          arrival_us=np.append(prob.arrival_us, 7), lat_us=np.append(prob.lat_us, np.full(D, 9, np.int32)),
                          peak_mib=np.append(prob.peak_mib, np.full(D, prob.weight_mib[0] + 1, np.int32)))
    prob = prob.with_(lat_us=np.minimum(prob.lat_us.astype(np.int64) * scale, 2**31 - 1).astype(np.int32))
    plans = wfgen.make_plans(prob, 300, 5, p_retain=0.7)
    plans.place[2, 0] = prob.D
    plans.order[4, 0] = plans.order[4, 1]
    out = wf.Results(plans.P)
    wf.wf_eval_plans_static(wf.DeviceProblem(prob), wf.DevicePlans.from_host(plans, "cuda"), out)
    wf.wf_static_status()
    want = oracle.eval_plans(prob, plans)
    if scale > 1:
        assert want[0][want[3] == 0].max() > 1 << 32
    for a, b in zip(out.numpy(), want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("D,M,scale", [(3, 4, 1), (7, 12, 1), (32, 16, 1), (2, 3, 1 << 20)])
def test_large_batches_of_short_windows(D, M, scale):
    """Batches around the one from which four warps share a CTA (16 plans an
    SM), the last CTA full and not, with and without retain rows, some invalid
    plans, and (the largest scale) run times that leave 32 bits."""
    import torch
    from randprob import random_problem
    from paper_2609_03335_gb300 import build, wf
    build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(40 + D)
    prob = random_problem(rng, n_sessions=4, sizes=(4, 12), D=D, M=M)
    prob = prob.with_(lat_us=np.minimum(prob.lat_us.astype(np.int64) * scale, 2**31 - 1).astype(np.int32))
    plans = wfgen.make_plans(prob, 16 * sms + 6, 5, p_retain=0.7 if D % 2 else None)
    plans.place[2, 0] = prob.D
    plans.order[4, 0] = plans.order[4, 1]
    want = oracle.eval_plans(prob, plans)
    dprob = wf.DeviceProblem(prob)
    for P in (16 * sms + 6, 16 * sms + 1, 16 * sms):
        out = wf.Results(P)
        wf.wf_eval_plans_static(dprob, wf.DevicePlans.from_host(plans.slice(0, P), "cuda"), out)
        wf.wf_static_status()
        for a, b in zip(out.numpy(), want):
            assert np.array_equal(a, b[:P])


@pytest.mark.parametrize("D,n,M,scale", [(1, 60, 1, 1), (2, 60, 5, 1), (2, 61, 5, 1), (3, 40, 9, 1), (4, 30, 3, 1), (4, 40, 3, 1), (4, 41, 3, 1),
                                         (4, 12, 4, 1 << 20)])
def test_large_batches_on_few_devices(D, n, M, scale):
    """Batches around the one from which short windows on up to four devices
    take a thread per plan (160 plans an SM), the longest such window and the
    next, in the static call and on the int64 path; retain rows, invalid plans,
    run times that leave 32 bits; and tables that fail the device check."""
    import torch
    from gpu_util import assert_same, gpu_eval
    from randprob import random_problem
    from paper_2609_03335_gb300 import build, wf
    build.build()
    most = 160 * torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(70 + n)
    prob = random_problem(rng, n_sessions=2, sizes=(n // 2, n - n // 2), D=D, M=M)
    while prob.N != n:
        prob = random_problem(rng, n_sessions=2, sizes=(n // 2, n - n // 2), D=D, M=M)
    prob = prob.with_(lat_us=np.minimum(prob.lat_us.astype(np.int64) * scale, 2**31 - 1).astype(np.int32))
    plans = wfgen.make_plans(prob, most + 1, 5, p_retain=0.7 if D % 2 else None)
    plans.place[2, 0] = prob.D
    plans.order[4, 0] = plans.order[4, 1]
    want = oracle.eval_plans(prob, plans, threads=8)
    dprob = wf.DeviceProblem(prob)
    for P in (most + 1, most):
        sub = plans.slice(0, P)
        out = wf.Results(P)
        wf.wf_eval_plans_static(dprob, wf.DevicePlans.from_host(sub, "cuda"), out)
        wf.wf_static_status()
        for a, b in zip(out.numpy(), want):
            assert np.array_equal(a, b[:P])
        assert_same(gpu_eval(prob, sub, int64_path=True), dict(zip(("makespan", "p95", "gpu", "status"), (w[:P] for w in want))))
    dprob.tensors["model"][n - 1] = M
    wf.wf_eval_plans_static(dprob, wf.DevicePlans.from_host(plans, "cuda"), out := wf.Results(most + 1))
    with pytest.raises(wf.WfError):
        wf.wf_static_status()
    assert (out.numpy()[3] == wf.ST_TABLES).all() and (out.numpy()[0] == wf.INT64_MAX).all()


@pytest.mark.parametrize("others", [[1] * 19, [1] * 3 + [0] * 16, [0] * 19, [3, 2, 1, 1, 0, 0], [1] * 250 + [2] * 60 + [0] * 5,
                                    [1] * 900 + [0] * 200])
def test_static_entry_with_sessions_that_own_no_activation(others):
    """Sessions that no activation belongs to, which the device check does not
    look for: their latency is INT64_MIN - arrival in wrapping 64-bit
    arithmetic (so INT64_MAX for an arrival of 1, the largest value there is),
    and the p95 is still the nearest rank of all sessions' values -- ranks near
    the top and, with many sessions, further down."""
    from randprob import random_problem
    from paper_2609_03335_gb300 import build, wf
    build.build()
    one = random_problem(np.random.default_rng(8), n_sessions=1, sizes=(6, 6), D=2, M=3).with_(arrival_us=np.zeros(1, np.int64))
    prob = one.with_(W=1 + len(others), arrival_us=np.r_[0, others].astype(np.int64))
    plans = wfgen.make_plans(one, 70, 4)
    mk, lat, gpu, st = oracle.eval_plans(one, plans)
    out = wf.Results(plans.P)
    wf.wf_eval_plans_static(wf.DeviceProblem(prob), wf.DevicePlans.from_host(plans, "cuda"), out)
    wf.wf_static_status()
    lo = np.full(len(others), np.iinfo(np.int64).min)
    with np.errstate(over="ignore"):
        none = lo - np.array(others, np.int64)
    assert (st == 0).all() and (1 not in others or none.max() == wf.INT64_MAX)
    rank = (95 * prob.W + 99) // 100 - 1
    want = np.sort(np.c_[np.tile(none, (plans.P, 1)), lat], axis=1)[:, rank]
    for a, b in zip(out.numpy(), (mk, want, gpu, st)):
        assert np.array_equal(a, b)
