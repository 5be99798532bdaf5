"""The stochastic sweep at its edges: sample counts around a warp's lanes, one
and two samples a lane and one to four timing warps a team; every model and
device count class; Box-Muller tables beyond 16 bits and too long for shared
memory.  Every result is a whole number, compared for equality."""
import numpy as np
import pytest

import wfgen
from gpu_util import assert_same, gpu_eval, oracle_eval
from randprob import random_problem
from test_gpu_parity import inject_invalid

pytestmark = pytest.mark.gpu


def tables(kind):
    r, c, e = wfgen.box_muller_tables()
    if kind == "wide":  # radii beyond 16 bits
        r = (r.astype(np.int64) * 3).astype(np.int32)
    elif kind == "long":  # more entries than shared memory takes
        r = np.tile(r, 16)
    zmax = -(-(int(np.abs(r).max()) * int(np.abs(c).max())) >> 18)
    e = np.rint(65536 * np.exp(0.2 * np.arange(-zmax, zmax + 1) / 256)).clip(0, 2**31 - 1).astype(np.int32)
    return r, c, e


@pytest.mark.parametrize("S,P,D,M,kind", [
    (1, 7, 1, 1, "short"), (32, 150, 3, 8, "short"), (33, 150, 8, 9, "short"), (64, 700, 12, 16, "short"),
    (65, 64, 4, 5, "short"), (127, 64, 4, 12, "short"), (129, 64, 32, 3, "short"), (200, 40, 5, 8, "short"),
    (256, 33, 2, 4, "short"), (257, 20, 2, 4, "short"), (64, 100, 3, 6, "wide"), (20, 100, 3, 10, "wide"),
    (100, 60, 3, 6, "long"), (16, 60, 3, 6, "long")])
def test_sample_counts_shapes_and_tables(S, P, D, M, kind):
    rng = np.random.default_rng(9000 + S + P)
    prob = random_problem(rng, n_sessions=5, D=D, M=M)
    r, c, e = tables(kind)
    prob = prob.with_(S=S, seed=int(rng.integers(0, 2**63)), bm_r=r, bm_c=c, bm_e=e)
    plans = wfgen.make_plans(prob, P, S, plan_base=int(rng.integers(0, 10**6)), p_retain=0.6 if S % 2 else None)
    if P >= 8:
        inject_invalid(plans, prob, rng)
    assert_same(gpu_eval(prob, plans), oracle_eval(prob, plans))


@pytest.mark.parametrize("S,P,D,M", [(20, 3000, 3, 4), (33, 2600, 9, 9), (64, 2500, 4, 5), (65, 2000, 5, 8), (129, 1500, 3, 10), (256, 1400, 2, 4)])
def test_teams_that_play_several_plans(S, P, D, M):
    """Short windows and enough plans that every team plays several in the same
    shared memory (at least one more than the chip holds at once), one and two
    samples a lane, one to four timing warps, invalid plans between the others."""
    rng = np.random.default_rng(9500 + S)
    prob = random_problem(rng, n_sessions=2, sizes=(5, 7), D=D, M=M)
    r, c, e = tables("short")
    prob = prob.with_(S=S, seed=int(rng.integers(0, 2**63)), bm_r=r, bm_c=c, bm_e=e)
    plans = wfgen.make_plans(prob, P, S, p_retain=0.6 if S % 2 else None)
    inject_invalid(plans, prob, rng)
    assert_same(gpu_eval(prob, plans), oracle_eval(prob, plans))
