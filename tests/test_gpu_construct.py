"""Bit-exact parity of the GPU plan constructor with the oracle's, and the
evaluator reproducing the constructor's timeline."""
import numpy as np
import pytest

import oracle
import wfgen
from gpu_util import lib
from randprob import random_problem

pytestmark = pytest.mark.gpu


def build(prob, P, seed, jitter, plan_base=0, retain=False):
    import torch
    wf = lib()
    ctx = wf.Ctx(prob, max_P=P)
    out = wf.DevicePlans.empty(P, prob.N, with_retain=retain, plan_base=plan_base)
    wf.wf_construct_plans(ctx, out, seed, jitter)
    res = wf.Results(P)
    wf.wf_eval_plans(ctx, out, res)
    torch.cuda.synchronize()
    wf.wf_ctx_status(ctx)
    return out.numpy(prob.N), res.numpy()


def check(prob, got, res, want, ends):
    for a, (g, w) in enumerate(zip(got[:4], (want.place, want.order, want.fuse, want.prefetch))):
        assert np.array_equal(g, w), ("field", a)
    mk, p95, gpu, st = res
    assert (st == 0).all()
    assert np.array_equal(mk, ends - int(np.min(prob.arrival_us)))


@pytest.mark.parametrize("case", range(6))
def test_random_windows(case):
    rng = np.random.default_rng(1500 + case)
    prob = random_problem(rng, n_sessions=int(rng.integers(1, 7)), D=int(rng.integers(1, 7)),
                          M=int(rng.integers(1, 7)))
    if case % 2:
        prob = prob.with_(grant_us=int(rng.integers(1, 500)))
    P = int(rng.integers(1, 200))
    jitter = [0, 1, 1000, 10 ** 6, 10 ** 9, 37][case]
    got, res = build(prob, P, seed=case, jitter=jitter, plan_base=17 * case, retain=case == 2)
    want, ends = oracle.construct(prob, P, seed=case, jitter=jitter, plan_base=17 * case)
    check(prob, got, res, want, ends)
    if case == 2:
        N = prob.N
        bits = np.unpackbits(got[4].view(np.uint8), bitorder="little", axis=1)[:, :N]
        assert bits.all() and not np.unpackbits(got[4].view(np.uint8), bitorder="little", axis=1)[:, N:].any()


@pytest.mark.parametrize("jitter", [2, 3, (1 << 40) + 12345, (1 << 46) - 1])
def test_jitter_remainders(jitter):
    """Jitter draws mod (jitter + 1) over the whole 64-bit range of the hash:
    the kernel's reciprocal-multiply remainder against the oracle's %."""
    rng = np.random.default_rng(77)
    prob = random_problem(rng, n_sessions=5, D=4, M=4)
    got, res = build(prob, 64, seed=9, jitter=jitter, plan_base=5)
    want, ends = oracle.construct(prob, 64, seed=9, jitter=jitter, plan_base=5)
    check(prob, got, res, want, ends)


@pytest.mark.parametrize("name,P", [("tiny", 300), ("mix", 200), ("burst", 64), ("large", 8)])
def test_named_workloads(name, P):
    prob = wfgen.config(name).problem
    got, res = build(prob, P, seed=5, jitter=200000, plan_base=3)
    want, ends = oracle.construct(prob, P, seed=5, jitter=200000, plan_base=3)
    check(prob, got, res, want, ends)


@pytest.mark.parametrize("D,M,P", [(1, 1, 1), (8, 8, 37), (8, 9, 5), (9, 16, 37), (16, 8, 3), (17, 8, 9), (32, 16, 5)])
def test_lanes_per_plan(D, M, P):
    """8, 16 and 32 lanes per plan, both queue words, and warps whose plans are not all there."""
    rng = np.random.default_rng(100 * D + M)
    prob = random_problem(rng, n_sessions=9, D=D, M=M)
    got, res = build(prob, P, seed=3, jitter=5000, plan_base=11)
    want, ends = oracle.construct(prob, P, seed=3, jitter=5000, plan_base=11)
    check(prob, got, res, want, ends)


@pytest.mark.parametrize("lengths,D,P", [([1], 1, 3), ([40], 3, 20000), ([25, 2], 12, 9000), ([12, 1, 1], 20, 5000)])
def test_the_last_ready_entry_is_taken(lengths, D, P):
    """Chains: the ready set holds one node or a few, so the node taken is often
    its last entry, whose place the next ready node takes at once -- over enough
    plans that every lane group builds a second one in the same scratch."""
    from test_gpu_edges import chains_window
    prob = chains_window(lengths, D=D, M=2, seed=len(lengths))
    got, res = build(prob, P, seed=2, jitter=300, plan_base=1)
    want, ends = oracle.construct(prob, P, seed=2, jitter=300, plan_base=1)
    check(prob, got, res, want, ends)


@pytest.mark.parametrize("D,M", [(5, 8), (8, 9), (13, 4), (16, 9)])
def test_lanes_by_batch(D, M):
    """The batches at which a plan takes 32, 16 or 8 lanes (12 and 24 plans an
    SM), and one more plan each, on one context made for the largest; the same
    seed gives the same plans whatever the lanes."""
    import torch
    wf = lib()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(D)
    prob = random_problem(rng, n_sessions=3, sizes=(4, 6), D=D, M=M)
    most = 24 * sms + 1
    ctx = wf.Ctx(prob, max_P=most)
    want, _ = oracle.construct(prob, most, seed=6, jitter=700)
    for P in (most, 24 * sms, 12 * sms + 1, 12 * sms, 3):
        out = wf.DevicePlans.empty(P, prob.N)
        wf.wf_construct_plans(ctx, out, 6, 700)
        torch.cuda.synchronize()
        wf.wf_ctx_status(ctx)
        for g, w in zip(out.numpy(prob.N)[:4], (want.place, want.order, want.fuse, want.prefetch)):
            assert np.array_equal(g, w[:P]), P
    ctx.close()
