"""What the certificates cost does not hang on a lane's spacing (needs a GB300).

The preparation is timed on lanes of the same vertex count: segments beyond a fixed length, or bends
beyond a fixed angle, must not make every certificate walk the whole lane.
"""
import statistics
import time

import numpy as np
import pytest
import torch

import paper_2308_01654_gb300 as mp
from paper_2308_01654_gb300 import scenarios as sc

pytestmark = pytest.mark.gpu


def prep_us(ref, **params):
    p = sc.default_params(512, 4, 0.05)
    p.update(**params)
    x0 = np.array([ref[0, 0], ref[0, 1], np.arctan2(*(ref[1] - ref[0])[::-1]), 7.0])
    with mp.Planner(p) as pl:
        pl.set_profiling(1)
        got = []
        for _ in range(40):
            pl.plan(x0, ref)
            got.append(pl.kernel_times()["prep"] * 1e3)
    return statistics.median(got[10:])


def bending(n, spacing, sigma):
    a = np.cumsum(np.random.default_rng(5).normal(0.0, sigma, n))
    return spacing * np.stack([np.cumsum(np.cos(a)), np.cumsum(np.sin(a))], 1)


# half a metre against one and three metres, straight, bending and in the vertex form: measured 1.0 times,
# and 2.7 to 3.7 times where long segments or bends are compared with the whole lane
@pytest.mark.parametrize("spacing", [1.0, 3.0])
@pytest.mark.parametrize("sigma,form", [(0.0, {}), (0.05, {}), (0.0, dict(ref_mode=1))])
def test_long_segments_and_bends_cost_no_more(spacing, sigma, form):
    base = prep_us(sc.straight_lane(4000, 0.5))
    assert prep_us(bending(4000, spacing, sigma), **form) < 1.6 * base


# a lane of 0.1 m spacing has five times the groups within reach: measured 0.95 times, and 1.5 to 1.6 times
# where each of their segments is compared
@pytest.mark.parametrize("lane", ["straight", "curved"])
def test_dense_lanes_cost_no_more(lane):
    make = sc.straight_lane if lane == "straight" else lambda n, d: sc.sinusoid_lane(n, d, 3.0, 80.0)
    assert prep_us(make(2000, 0.1)) < 1.25 * prep_us(make(2000, 0.5))


def device_us(n_ref, K=8192, T=100):
    p = sc.default_params(K, T, 0.05)
    stream = torch.cuda.Stream()
    x0, ref = (torch.tensor(a, dtype=torch.float64, device="cuda")
               for a in (np.array([0.0, 0.3, 0.0, 8.0]), sc.straight_lane(n_ref, 0.5)))
    u, x = (torch.empty(s, dtype=torch.float64, device="cuda") for s in ((T, 2), (T + 1, 4)))
    torch.cuda.synchronize()
    got = []
    with mp.Planner(p, stream=stream.cuda_stream) as pl:
        for _ in range(8):
            t = time.perf_counter()
            for _ in range(50):
                pl.plan_device(x0, ref, None, None, u, x)
            torch.cuda.synchronize()
            got.append((time.perf_counter() - t) / 50 * 1e6)
    return statistics.median(got[2:])


def test_certificates_do_not_pack_the_rollout():
    """The same rollouts on a longer lane: measured 1.04 times, and 1.25 where the rollout's blocks are
    placed two to an SM beside the SMs that still form certificates."""
    assert device_us(1000) < 1.14 * device_us(200)


# both triggers, and both sides of the rule between them (blocks of 128 threads and of 160, one to an SM and
# more), give the same bits
@pytest.mark.parametrize("K,group,block", [(512, -16, 128), (512, -16, 160), (152 * 128, 1, 128),
                                           (152 * 128 + 1, 1, 128), (4864, -8, 448)])
@pytest.mark.parametrize("n_ref", [3, 700])
def test_the_trigger_changes_no_bit(K, group, block, n_ref):
    p = sc.default_params(K, 9, 0.05)
    got = []
    for shape in (dict(group=group, block=block), dict(group=1, block=64)):
        with mp.Planner(dict(p, **shape)) as pl:
            for _ in range(3):
                u, x, info = pl.plan(np.array([0.0, 0.3, 0.1, 8.0]), sc.sinusoid_lane(n_ref, 0.5, 3.0, 80.0))
            got.append((u, x, pl.get_costs(), info))
    for a, b in zip(got[0][:3], got[1][:3]):
        np.testing.assert_array_equal(a, b)
    assert got[0][3] == got[1][3]
