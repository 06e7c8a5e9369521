"""Two and four lanes splitting the work of each step take the specialised rollout step (needs a GB300).

Same bits as one lane per sample, on both sides of the broad phase's one pass of 32 circles, and faster
than the general step, which eight lanes take.
"""
import statistics

import numpy as np
import pytest

import paper_2308_01654_gb300 as mp
from paper_2308_01654_gb300 import scenarios as sc

pytestmark = pytest.mark.gpu


def scene(n_obs, **params):
    p = sc.default_params(params.pop("K", 777), params.pop("T", 15), 0.05)
    p.update(**params)
    ref = sc.straight_lane(400, 0.5)
    rng = np.random.default_rng(n_obs)
    circ = sc.obstacle_circles(rng, ref, n_obs, (5.0, 60.0), (-3.0, 3.0)) if n_obs else np.zeros((0, 5))
    return p, np.array([0.0, 0.3, 0.1, 8.0]), ref, circ


@pytest.mark.parametrize("n_obs", [0, 3, 10, 11, 40])
@pytest.mark.parametrize("group,block", [(2, 64), (4, 128), (4, 896)])
@pytest.mark.parametrize("bf16", [0, 1])
def test_the_same_bits(n_obs, group, block, bf16):
    got = []
    for shape in (dict(group=group, block=block), dict(group=1, block=64)):
        p, x0, ref, circ = scene(n_obs, noise_bf16=bf16, **shape)
        with mp.Planner(p) as pl:
            u, x, info = pl.plan(x0, ref, circ)
            got.append((u, x, pl.get_costs(), info))
    for a, b in zip(got[0][:3], got[1][:3]):
        np.testing.assert_array_equal(a, b)
    assert got[0][3] == got[1][3]


def rollout_us(group):
    p, x0, ref, circ = scene(32, K=8192, T=100, group=group, block=128)
    with mp.Planner(p) as pl:
        pl.set_profiling(1)
        us = []
        for _ in range(30):
            pl.plan(x0, ref, circ)
            us.append(pl.kernel_times()["rollout"] * 1e3)
    return statistics.median(us[10:])


# measured 0.60 of the general step's time with eight lanes, and 0.86 to 0.88 where two and four lanes run the general
# step as well
@pytest.mark.parametrize("group", [2, 4])
def test_the_specialised_step_runs(group):
    assert rollout_us(group) < 0.74 * rollout_us(8)
