"""The launch rules and the variants they choose (needs a GB300): none of them changes a result.

The lanes per sample, the block size, the graph and the steps per tile of the weighted sum follow from
the sizes; each result here is compared with the same plan under a fixed plain shape (one lane per
sample), and the specialised step, the vertex window and the clustered cost-to-go weights with the
oracle, at the edges of their windows and runs (up to two of 2048 samples may pass within 1e-5 m of a
cost jump and miss the cost tolerance, the rule of parity.py).
"""
import numpy as np
import pytest

import oracle
import paper_2308_01654_gb300 as mp
from paper_2308_01654_gb300 import scenarios as sc
from parity import assert_costs, assert_update

pytestmark = pytest.mark.gpu


def turned(prob, angle=0.7, shift=(150.0, -80.0)):
    """The scene turned and moved in the plane (headings of a straight lane then differ in their last bits)."""
    c, s = np.cos(angle), np.sin(angle)
    R, o = np.array([[c, s], [-s, c]]), np.array(shift)
    q = prob.copy()
    q.ref = q.ref @ R + o
    if q.circles.size:
        q.circles[:, :2] = q.circles[:, :2] @ R + o
        q.circles[:, 3:] = q.circles[:, 3:] @ R
    q.x0[:2] = q.x0[:2] @ R + o
    q.x0[2] += angle
    return q


def small(K, T, n_ref=120, lane="straight", n_obs=3, **params):
    p = sc.default_params(K, T, 0.05)
    p.update(seed=K + T, **params)
    ref = sc.straight_lane(n_ref, 0.5) if lane == "straight" else sc.sinusoid_lane(n_ref, 0.5, 3.0, 80.0)
    rng = np.random.default_rng(K)
    circ = sc.obstacle_circles(rng, ref, n_obs, (5.0, 40.0), (-3.0, 3.0)) if n_obs else np.zeros((0, 5))
    yaw = float(np.arctan2(*(ref[1] - ref[0])[::-1]))
    return turned(sc.Problem(p, np.array([0.0, 0.3, yaw, 8.0]), ref, circ))


def plan(prob, **shape):
    prob = prob.copy()
    prob.params.update(**shape)
    with mp.Planner(prob.params) as pl:
        u, x, info = pl.plan(prob.x0, prob.ref, prob.circles, prob.centres)
        return u, x, info, pl.get_costs()


# one warp's worth, both sides of each change of split (16, 8, 4, 2 and 1 lanes), odd sizes
@pytest.mark.parametrize("K,T", [(1, 1), (31, 3), (300, 17), (4256, 20), (4257, 9), (17025, 8), (34049, 5),
                                 (68097, 4), (140001, 2)])
@pytest.mark.parametrize("lane", ["straight", "curved"])
def test_chosen_shape_gives_the_one_lane_costs(K, T, lane):
    prob = small(K, T, lane=lane)
    a, b = plan(prob), plan(prob, group=1, block=128)
    np.testing.assert_array_equal(a[3], b[3])
    np.testing.assert_array_equal(a[0], b[0])
    assert a[2] == b[2]


# circles: none, up to one pass of the broad phase, and past it (bucket range)
@pytest.mark.parametrize("n_obs", [0, 1, 10, 11, 30])
@pytest.mark.parametrize("n_ref", [2, 3, 4, 513, 1026])
def test_specialised_step_against_the_oracle(n_obs, n_ref):
    prob = small(2048, 12, n_ref=n_ref, n_obs=n_obs)
    u, x, info, S = plan(prob)
    orc = oracle.plan(prob)
    assert_costs(S, orc.S, orc.margin, max_excused_fail=1e-3)
    assert_update(u, x, orc)


@pytest.mark.parametrize("n_ref", [2, 3, 60, 1025])
def test_vertex_window_against_the_oracle(n_ref):
    prob = small(2048, 12, n_ref=n_ref, lane="curved", ref_mode=1)
    u, x, info, S = plan(prob)
    orc = oracle.plan(prob)
    assert_costs(S, orc.S, orc.margin, max_excused_fail=1e-3)
    assert_update(u, x, orc)


# runs of the clustered weights: one block, its edges, and the most blocks
@pytest.mark.parametrize("K", [1, 255, 2048, 2049, 8193])
def test_cost_to_go_weights_against_the_oracle(K):
    prob = small(K, 6, cost_to_go=1)
    u, x, info, S = plan(prob)
    orc = oracle.plan(prob)
    assert_costs(S, orc.S, orc.margin)
    assert_update(u, x, orc)


# steps per tile of the weighted sum: every length the rule takes, binary32 and bfloat16 noise
@pytest.mark.parametrize("K,T", [(2048, 40), (65536, 60), (65536, 100), (65536, 200), (131072, 90)])
@pytest.mark.parametrize("bf16", [0, 1])
def test_update_is_the_sum_over_the_noise(K, T, bf16):
    prob = small(K, T, n_obs=0, noise_bf16=bf16, sg_enable=0, sigma=[0.2, 0.01], u_min=[-9.0, -0.5], u_max=[9.0, 0.5])
    with mp.Planner(prob.params) as pl:
        u, x, info = pl.plan(prob.x0, prob.ref, prob.circles)
        S, z = pl.get_costs(), pl.get_noise().astype(np.float64)
    w = np.exp(-(S - S.min()) / prob.params["lam"])
    want = np.stack([np.einsum("k,tk->t", w, z[:, :, c]) * prob.params["sigma"][c] for c in (0, 1)], 1) / w.sum()
    # binary32 weights (a few 1e-7 times the exponent) and binary32 partial sums of 256 products
    np.testing.assert_allclose(u, want, rtol=0, atol=2e-6)


# one plan to several, lanes per sample 16 .. 1
@pytest.mark.parametrize("sizes", [[257], [4096, 300], [20000, 16384, 2048], [65536, 30000, 5]])
def test_batch_rule_gives_the_one_lane_results(sizes):
    probs = [small(K, 7 + 3 * i, lane=("straight", "curved")[i % 2], n_obs=(2, 12, 0)[i % 3], session=i)
             for i, K in enumerate(sizes)]
    caps = dict(max_slots=8, max_batch=8, max_samples=sum(sizes), max_rollout_steps=sum(p.K * p.T for p in probs),
                max_T=32, max_ref=256, max_circ=64)
    got = []
    for fixed in (False, True):
        with mp.BatchPlanner(**caps) as bp:
            if fixed:
                bp.set_launch(1, 128)
            plans = [mp.BatchPlan(p.params, i, p.x0, p.ref, p.circles) for i, p in enumerate(probs)]
            bp.plan(plans)
            got.append([(p.u.copy(), p.x.copy(), p.info.as_dict()) for p in plans])
    for a, b in zip(*got):
        np.testing.assert_array_equal(a[0], b[0])
        np.testing.assert_array_equal(a[1], b[1])
        assert a[2] == b[2]
