"""Tuning a batch planner on a small submission does not lose to the library's own rule (needs a GB300).

For small submissions the rule splits the steps among 16 lanes, a shape that a caller cannot set: tuning
times it too, keeps it where it is the fastest, and reports a shape that can be set.
"""
import statistics
import time

import numpy as np
import pytest

import paper_2308_01654_gb300 as mp
from paper_2308_01654_gb300 import scenarios as sc

pytestmark = pytest.mark.gpu


def planner_and_plans(sizes, T):
    plans = []
    for i, K in enumerate(sizes):
        p = sc.default_params(K, T, 0.05)
        p.update(session=i)
        plans.append(mp.BatchPlan(p, i, np.array([0.0, 0.3, 0.0, 8.0]), sc.straight_lane(300, 0.5), np.zeros((0, 5))))
    bp = mp.BatchPlanner(max_slots=8, max_batch=8, max_samples=sum(sizes), max_rollout_steps=sum(sizes) * T, max_T=T,
                         max_ref=300, max_circ=4)
    return bp, plans


def median_us(bp, plans):
    reqs, got = bp.requests(plans), []
    for _ in range(60):
        t = time.perf_counter()
        bp.plan(plans, reqs)
        got.append((time.perf_counter() - t) * 1e6)
    return statistics.median(got[20:])


@pytest.mark.parametrize("sizes", [[300], [1024], [2048, 1500], [12000]])
def test_the_reported_shape_can_be_set_and_the_results_stay(sizes):
    out = []
    for tune in (False, True):
        bp, plans = planner_and_plans(sizes, 20)
        with bp:
            if tune:
                g, b = bp.autotune(plans)
            bp.plan(plans)
            out.append([(p.u.copy(), p.x.copy(), p.info.as_dict()) for p in plans])
            if tune:
                bp.set_launch(g, b)
    for a, b in zip(*out):
        np.testing.assert_array_equal(a[0], b[0])
        np.testing.assert_array_equal(a[1], b[1])
        assert a[2] == b[2]


# measured 1.00 times the untuned planner, and 1.11 to 1.21 where tuning cannot choose the rule's 16 lanes
@pytest.mark.parametrize("sizes", [[2048], [4096]])
def test_tuning_is_not_slower_than_the_rule(sizes):
    bp, plans = planner_and_plans(sizes, 150)
    with bp:
        rule = median_us(bp, plans)
        bp.autotune(plans)
        assert median_us(bp, plans) < 1.05 * rule
