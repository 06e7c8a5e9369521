"""Lanes that meet themselves, with the rollouts exactly on the meeting point (needs a GB300).

The closest segment (or vertex) is the one of the smallest distance and, among equal distances, the
lowest index, whichever branch of the lane the rollout came along.  The vehicle stands a quarter of a
metre before the meeting point and reaches it in one step without rounding, so both branches are at
distance zero there and the cost tells which one was taken (their headings differ).
"""
import numpy as np
import pytest

import oracle
import paper_2308_01654_gb300 as mp
from paper_2308_01654_gb300 import scenarios as sc
from parity import assert_costs, assert_update

pytestmark = pytest.mark.gpu


def leg(a, b):
    """Vertices from a (included) to b (left out), half a metre apart."""
    a, b = np.array(a, float), np.array(b, float)
    n = int(round(np.abs(b - a).max() / 0.5))
    return a + (b - a) * (np.arange(n) / n)[:, None]


def crossing(at_vertex):
    """North past x = 0.25, around to the left, and east along y = 0 over itself, in the middle of two
    segments or at a vertex of each."""
    y, x = (0.0, -9.75) if at_vertex else (0.25, -10.0)
    return np.concatenate([leg((0.25, y - 10.0), (0.25, y + 10.0)), leg((0.25, y + 10.0), (x, y + 10.0)),
                           leg((x, y + 10.0), (x, 0.0)), leg((x, 0.0), (x + 25.0, 0.0))])


def ring():
    """A square whose last vertex is its first."""
    c = [(0.25, 0.0), (0.25, 10.0), (-9.75, 10.0), (-9.75, 0.0), (0.25, 0.0)]
    return np.concatenate([leg(a, b) for a, b in zip(c, c[1:])] + [np.array(c[-1:])])


LANES = {"middle": lambda: crossing(False), "vertex": lambda: crossing(True), "ring": ring}


def problem(ref, T, **params):
    p = sc.default_params(64, T, 0.0625)
    p.update(**params)
    return sc.Problem(p, np.array([0.0, 0.0, 0.0, 4.0]), ref, np.zeros((0, 5)))


# one lane per sample, steps and work split among lanes; the vertex form; the general step (a speed cap)
@pytest.mark.parametrize("shape", [dict(group=1, block=64), dict(group=-2, block=64), dict(group=-16, block=64),
                                   dict(group=8, block=64)])
@pytest.mark.parametrize("form", [dict(), dict(ref_mode=1), dict(v_max=9.0)])
@pytest.mark.parametrize("name", list(LANES))
def test_a_meeting_point_belongs_to_the_lowest_index(name, form, shape):
    if name == "middle" and "ref_mode" in form:
        pytest.skip("no vertex at the meeting point")
    prob = problem(LANES[name](), 1, **form, **shape)
    with mp.Planner(prob.params) as pl:
        u, x, _ = pl.plan(prob.x0, prob.ref, prob.circles)
        S = pl.get_costs()
    orc = oracle.plan(prob)
    assert orc.S.min() > 100.0          # the first branch: the vehicle is at right angles to it
    assert_costs(S, orc.S, orc.margin)
    assert_update(u, x, orc)


def test_a_meeting_point_in_a_batch():
    probs = [problem(make(), 1, session=i) for i, make in enumerate(LANES.values())]
    with mp.BatchPlanner(max_slots=4, max_batch=4, max_samples=256, max_rollout_steps=256, max_T=4, max_ref=256,
                         max_circ=4) as bp:
        plans = [mp.BatchPlan(p.params, i, p.x0, p.ref, p.circles) for i, p in enumerate(probs)]
        reqs = bp.requests(plans)
        ticket = bp.submit(reqs)
        bp.wait(ticket)
        for i, p in enumerate(probs):
            orc = oracle.plan(p)
            assert_costs(bp.get_costs(ticket, i, p.K), orc.S, orc.margin)
