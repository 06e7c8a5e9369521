"""The weighted sum in tiles of every length its rule takes (needs a GB300).

The update is recomputed from the planner's own costs and noise; with cost-to-go weights it is compared
with the oracle.
"""
import numpy as np
import pytest

import oracle
import paper_2308_01654_gb300 as mp
from paper_2308_01654_gb300 import scenarios as sc
from parity import assert_update

pytestmark = pytest.mark.gpu

# (samples, steps) that take tiles of 1, 2, 3, 4, 6 and 8 steps on 152 SMs
PLAIN = [(2048, 40), (65536, 50), (65536, 90), (65536, 128), (65536, 200), (374784, 40)]
STAGED = [(2048, 40), (65536, 50), (65536, 90), (178176, 40)]          # bfloat16 noise, rows of 16 bytes
CTG = [(65536, 100), (65536, 128), (65536, 200)]


def problem(K, T, **params):
    p = sc.default_params(K, T, 0.05)
    p.update(seed=K + T, **params)
    return sc.Problem(p, np.array([0.0, 0.3, 0.0, 8.0]), sc.straight_lane(20, 10.0), np.zeros((0, 5)))


@pytest.mark.parametrize("K,T,bf16", [(K, T, 0) for K, T in PLAIN] + [(K + 2, T, 1) for K, T in PLAIN] +
                         [(K, T, 1) for K, T in STAGED])
def test_update_is_the_sum_over_the_noise(K, T, bf16):
    prob = problem(K, T, noise_bf16=bf16, sg_enable=0, sigma=[0.2, 0.01], u_min=[-9.0, -0.5], u_max=[9.0, 0.5])
    with mp.Planner(prob.params) as pl:
        u, x, info = pl.plan(prob.x0, prob.ref, prob.circles)
        S, z = pl.get_costs(), pl.get_noise()
    w = np.exp(-(S - S.min()) / prob.params["lam"])
    keep = np.nonzero(w)[0]
    want = np.stack([np.einsum("k,tk->t", w[keep], z[:, keep, c].astype(np.float64)) * prob.params["sigma"][c]
                     for c in (0, 1)], 1) / w.sum()
    # binary32 weights (a few 1e-7 times the exponent) and binary32 partial sums of 256 products
    np.testing.assert_allclose(u, want, rtol=0, atol=2e-6)


@pytest.mark.parametrize("K,T", CTG)
def test_cost_to_go_update_against_the_oracle(K, T):
    prob = problem(K, T, cost_to_go=1)
    with mp.Planner(prob.params) as pl:
        u, x, _ = pl.plan(prob.x0, prob.ref, prob.circles)
    assert_update(u, x, oracle.plan(prob))
