"""Groups of segments that the certificates pass over unseen (no GPU).

A certificate of the closest-point search is computed against every other segment, in groups of 32; a
group is passed over when that cannot change the result.  The rules are restated in numpy and checked on
lanes of short and long, even and uneven segments, folded over themselves or not.
"""
import numpy as np
import pytest

from test_search_bound import F

CAP, FAR, LONG = 12.0, 30.0, 1e3
GROUP = 32


def lane(rng, kind, spacing, n=400):
    """A polyline in binary32."""
    ln = spacing * (rng.uniform(0.97, 1.03, n - 1) if kind != "uneven" else np.exp(rng.normal(0.0, 1.0, n - 1)))
    ang = rng.uniform(-np.pi, np.pi) + {"straight": np.zeros(n - 1), "bends": 0.3 * np.sin(np.arange(n - 1) / 9.0),
                                        "uneven": np.cumsum(rng.normal(0.0, 0.02, n - 1)),
                                        "sharp": np.cumsum(rng.normal(0.0, 0.5, n - 1)),
                                        "there_and_back": np.where(np.arange(n - 1) < n // 2, 0.0, np.pi - 1e-3)}[kind]
    w = np.zeros((n, 2))
    w[0] = rng.uniform(-300.0, 300.0, 2)
    w[1:] = w[0] + np.cumsum(ln[:, None] * np.stack([np.cos(ang), np.sin(ang)], 1), 0)
    return w.astype(F)


def groups(v):
    """Per group of 32 segments: its first and last vertex, bounding circle and longest segment."""
    out = []
    for j0 in range(0, len(v) - 1, GROUP):
        p = v[j0:j0 + GROUP + 1]
        lo, hi = p.min(0), p.max(0)
        h = (F(0.5) * (hi - lo)).astype(F)
        rho = F(1.001) * np.sqrt((h * h).sum()).astype(F) + F(1e-3)
        l2 = ((p[1:] - p[:-1]) ** 2).sum(1).max()
        out.append((j0, j0 + len(p) - 1, lo + h, rho, l2))
    return out


def passed_far(v, i, g, vertex):
    """The rule by distance, for the item that starts at vertex i."""
    ln = F(np.hypot(*(v[i + 1] - v[i]))) if i + 1 < len(v) else F(0)
    reach = F(FAR) + (F(0) if vertex else ln) + g[3]
    d = g[2] - v[i]
    return bool(ln <= LONG and (d * d).sum() >= reach * reach and g[4] <= LONG * LONG)


def point_segment(p, a, b):
    p, a, b = (np.asarray(u, np.float64) for u in (p, a, b))
    e = b - a
    l2 = (e * e).sum(-1)
    t = np.clip(((p - a) * e).sum(-1) / np.where(l2 > 0, l2, 1.0), 0.0, 1.0)
    return np.hypot(*np.moveaxis(p - a - t[..., None] * e, -1, 0))


def gap(v, i, j0, j1, vertex):
    """Distance from the item at i (segment or vertex) to the segments j0 .. j1 - 1, none crossing it."""
    a, b = v[j0:j1], v[j0 + 1:j1 + 1]
    d = point_segment(v[i], a, b).min()
    if not vertex:
        d = min(d, point_segment(v[i + 1], a, b).min(), point_segment(a, v[i], v[i + 1]).min(),
                point_segment(b, v[i], v[i + 1]).min())
    return d


KINDS = ["straight", "bends", "uneven", "sharp", "there_and_back"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("spacing", [0.1, 0.5, 1.0, 5.0, 40.0])
@pytest.mark.parametrize("vertex", [False, True])
def test_a_group_passed_by_distance_is_out_of_reach(kind, spacing, vertex):
    """A point within CAP of the item is then closer to it than to the group by 0.4 CAP and more."""
    rng = np.random.default_rng([KINDS.index(kind), int(10 * spacing)])
    v = lane(rng, kind, spacing)
    gs, passed = groups(v), 0
    for i in range(0, len(v) - 1, 7):
        for g in gs:
            if passed_far(v, i, g, vertex):
                assert gap(v, i, g[0], g[1], vertex) >= 2.4 * CAP
                passed += 1
    if kind == "straight" and spacing >= 0.5:         # most of the lane lies beyond the reach
        assert passed > 0.4 * len(range(0, len(v) - 1, 7)) * len(gs)


def test_the_rule_holds_the_kernels_constants():
    import os
    import re
    src = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_01654_gb300",
                            "csrc", "mppi_iter.cuh")).read()
    const = {k: eval(v.replace("f", "").replace("CERT_CAP", "12.0"))
             for k, v in re.findall(r"constexpr float (CERT_\w+) = ([^;]+);", src)}
    assert const == {"CERT_CAP": CAP, "CERT_FAR": FAR, "CERT_LONG": LONG}
