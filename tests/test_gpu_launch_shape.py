"""The walk's launch shape follows the number of walkers (warps per CTA and CTAs, up to a full
GPU): the trajectories do not depend on it."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import paper_2011_00068_gb300 as labs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,kw", [(41, {}), (201, {}), (401, {}), (151, {"objective": "psl"}), (101, {"flags": 32})])
@pytest.mark.parametrize("walkers", [1, 151, 609, 1217, 2433, 4000])
def test_walkers_do_not_depend_on_the_launch_shape(L, kw, walkers):
    out = []
    for shape in ({}, {"warps_per_cta": 8}, {"warps_per_cta": 1}):
        s = labs.Search(L, walkers, 5, chunk_steps=20, **shape, **kw)
        s.walk(48)
        out.append(s.results(seqs=True))
        s.close()
    for k in ("isl", "best_isl", "seq", "best_seq"):
        assert np.array_equal(out[0][k], out[1][k]) and np.array_equal(out[0][k], out[2][k]), k
    if not kw:
        o = oracle.walk(L, 5, min(walkers, 40), 48)
        assert np.array_equal(out[0]["isl"][:40], o["final_isl"])
        assert np.array_equal(out[0]["best_seq"][:40], o["best_seq"])


@pytest.mark.parametrize("L,walkers", [(513, 1), (601, 153), (513, 640)])
def test_long_walkers_on_as_many_ctas(L, walkers):
    s = labs.Search(L, walkers, 5, chunk_steps=5)
    s.walk(12)
    r = s.results(seqs=True)
    s.close()
    o = oracle.walk(L, 5, min(walkers, 6), 12)
    assert np.array_equal(r["isl"][:6], o["final_isl"])
    assert np.array_equal(r["seq"][:6], o["final_seq"])


@pytest.mark.parametrize("L,many", [(41, 1300), (101, 700), (151, 700), (201, 400), (401, 150)])
@pytest.mark.parametrize("kw", [{}, {"tabu_log2": 4, "probe_cap": 3}, {"tabu_log2": 5, "probe_cap": 1},
                                {"tabu_log2": 6, "probe_cap": 32, "patience": 30}, {"tabu_log2": 3, "probe_cap": 20}])
def test_few_and_many_walkers_take_the_same_steps(L, many, kw):
    """Few walkers look every neighbour up at a step's start, many the lowest two: the first
    walkers of both searches, and the oracle's, agree step for step, also where HT is nearly
    full, single slots are probed or every state is taken."""
    few, steps, got = 9, 90, []
    for W in (few, many):
        s = labs.Search(L, W, 11, **kw)
        code, isl = s.trace(list(range(few)), steps)
        s.walk(steps)
        s.sync()
        r = s.results(seqs=True)
        got.append((code.cpu().numpy(), isl.cpu().numpy(), r["isl"][:few], r["best_isl"][:few], r["seq"][:few]))
        s.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    o = oracle.walk(L, 11, few, steps, trace=True, **kw)
    assert np.array_equal(got[0][0], o["trace_code"]) and np.array_equal(got[0][1], o["trace_isl"])
    assert np.array_equal(got[0][4], o["final_seq"])
