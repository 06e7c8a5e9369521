"""Circles sorted along either coordinate axis (needs a GB300).

The order only narrows the broad phase: costs agree with the oracle for static, moving and tabulated
circles on lanes of any heading, on both sides of one pass of 32 circles.
"""
import numpy as np
import pytest

import oracle
import paper_2308_01654_gb300 as mp
from paper_2308_01654_gb300 import scenarios as sc
from parity import assert_costs, assert_update

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33])
@pytest.mark.parametrize("angle", [0.0, 0.8, 1.5707963, 2.5, -2.0])
@pytest.mark.parametrize("motion", ["static", "moving", "table"])
def test_costs_against_the_oracle(n, angle, motion):
    p = sc.default_params(1024, 10, 0.05)
    p.update(seed=n)
    rng = np.random.default_rng(n)
    c, s = np.cos(angle), np.sin(angle)
    R, o = np.array([[c, s], [-s, c]]), np.array([120.0, -60.0])
    ref = sc.straight_lane(150, 0.5) @ R + o
    circ = np.zeros((n, 5))
    circ[:, 0], circ[:, 1], circ[:, 2] = rng.uniform(-2.0, 25.0, n), rng.uniform(-6.0, 6.0, n), rng.uniform(0.5, 1.2, n)
    if motion != "static":
        circ[:, 3:] = rng.uniform(-8.0, 8.0, (n, 2))
    circ[:, :2], circ[:, 3:] = circ[:, :2] @ R + o, circ[:, 3:] @ R
    t = (np.arange(10) + 1.0)[:, None, None] * 0.05
    centres = np.ascontiguousarray(circ[None, :, :2] + circ[None, :, 3:] * t) if motion == "table" else None
    prob = sc.Problem(p, np.concatenate([np.array([0.0, 0.3]) @ R + o, [angle, 8.0]]), ref, circ, centres)
    with mp.Planner(p) as pl:
        u, x, _ = pl.plan(prob.x0, prob.ref, prob.circles, prob.centres)
        S = pl.get_costs()
    orc = oracle.plan(prob)
    assert_costs(S, orc.S, orc.margin, max_excused_fail=1e-3)
    assert_update(u, x, orc)
