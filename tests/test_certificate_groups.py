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


def unit(d):
    d = np.asarray(d, np.float64)
    ln = np.hypot(*d)
    return (d / ln, ln) if ln > 0 else (d, 0.0)


def item(v, i):
    """The segment form's item at i: origin, direction, length, sines and outsides of the leans, least gap."""
    v = v.astype(np.float64)
    t, ln = unit(v[i + 1] - v[i])
    nxt = unit(v[i + 2] - v[i + 1]) if i + 2 < len(v) else None
    prv = unit(v[i - 1] - v[i]) if i > 0 else None
    lens = [ln] + [u[1] for u in (nxt, prv) if u]
    lmin, lmax = min(lens), max(lens)
    om = np.sqrt(2.0 ** -19 * (1 + 4 * lmax / lmin)) + 2.0 ** -20 * (CAP + lmax) / lmin + 2e-6
    sp = sm = 1.0
    op = od = 0.0
    if nxt and t @ nxt[0] > 0:
        c = t[0] * nxt[0][1] - t[1] * nxt[0][0]
        sp, op = min(abs(c) + om, 1.0), -1.0 if c > 0 else 1.0
    if prv and t @ prv[0] < 0:
        c = t[0] * prv[0][1] - t[1] * prv[0][0]
        sm, od = min(abs(c) + om, 1.0), -1.0 if c > 0 else 1.0
    return v[i], t, ln, sp, sm, op, od, min(om, 1.0), 0.55 * lmin + 2.0 ** -18 * lmax


def in_frame(it, p):
    w = np.asarray(p, np.float64) - it[0]
    return w @ it[1], w @ np.array([-it[1][1], it[1][0]])


def roots(it, a, b):
    """The certificate's distance against each segment a-b, the better of its two bounds."""
    _, _, ln, sp, sm, op, od, om, gap_ = it
    (ax, ay), (bx, by) = in_frame(it, a), in_frame(it, b)
    fwd, bwd = np.minimum(ax, bx) - ln, -np.maximum(ax, bx)
    gx, ahead = np.maximum(np.maximum(fwd, bwd), 0.0), fwd > bwd
    s = np.where(gx > 0, np.where(ahead, sp, sm), max(sp, sm))
    o = np.where(ahead, op, od)
    yn = np.where(np.where(ahead, ax <= bx, ax >= bx), ay, by)
    ymax = np.maximum(abs(ay), abs(by))
    ymin = np.where(ay * by <= 0, 0.0, np.minimum(abs(ay), abs(by)))
    dxj = abs(bx - ax)
    lj = np.maximum(ln, dxj + abs(by - ay))
    c2, bl, qa = 2.0 ** -37 * lj * lj, 1.016 * 2.0 ** -19 * lj, 1.016 * 2.0 ** -18
    n1, n2 = gx * gx + ymin * ymin - c2, gx * gx - c2
    nn = np.maximum(yn + gx * np.where(o >= 0, s, om), -yn + gx * np.where(o <= 0, s, om))
    b1, b2, a1 = ymax + gx * s + bl, np.maximum(nn, 0.0) + bl, s * s + qa
    with np.errstate(all="ignore"):
        r1 = n1 / (b1 + np.sqrt(b1 * b1 + a1 * np.maximum(n1, 0)))
        r2 = np.minimum(n2 / (b2 + np.sqrt(b2 * b2 + qa * np.maximum(n2, 0))), gx * dxj / (s * dxj + abs(by - ay)))
    r = np.maximum(np.where(n1 > 0, r1, 0.0), np.where((n2 > 0) & (dxj > 0), r2, 0.0))
    return np.where(gx * gx + ymin * ymin >= gap_ * gap_, r, 0.0)


def passed_thick(v, it, j0, j1, l2):
    """The rule for a group as one thick segment."""
    a, b = v[j0].astype(np.float64), v[j1].astype(np.float64)
    h = 1.001 * point_segment(v[j0:j1 + 1], a, b).max() + 1e-4 + 2.0 ** -18 * np.abs(b - a).sum() / 2
    _, _, ln, sp, sm, _, _, _, gap_ = it
    (ax, ay), (bx, by) = in_frame(it, a), in_frame(it, b)
    fwd, bwd = min(ax, bx) - ln, -max(ax, bx)
    gx, s = max(fwd, bwd) - h, sp if fwd > bwd else sm
    ymax = max(abs(ay), abs(by)) + h
    ymin = 0.0 if ay * by <= 0 else max(min(abs(ay), abs(by)) - h, 0.0)
    l = max(ln, 1.5 * np.sqrt(l2))
    g2, b1, a1 = gx * gx + ymin * ymin, ymax + gx * s + 1.016 * 2.0 ** -19 * l, s * s + 1.016 * 2.0 ** -18
    return (gx >= CAP * s and gx > 0 and g2 >= gap_ * gap_ and
            g2 - 2.0 ** -37 * l * l >= CAP * (a1 * CAP + 2 * b1))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("spacing", [0.02, 0.1, 0.5, 5.0, 40.0])
def test_no_segment_of_a_group_passed_as_one_lowers_the_certificate(kind, spacing):
    rng = np.random.default_rng([KINDS.index(kind), int(100 * spacing), 2])
    v = lane(rng, kind, spacing, 800)
    gs, passed = groups(v), 0
    for i in range(0, len(v) - 1, 13):
        it = item(v, i)
        for j0, j1, _, _, l2 in gs:
            if (i + 1 < j0 or i - 1 >= j1) and passed_thick(v, it, j0, j1, l2):
                assert roots(it, v[j0:j1], v[j0 + 1:j1 + 1]).min() >= CAP
                passed += 1
    if kind in ("straight", "bends"):                 # the lanes it is for
        assert passed > 0


def test_the_rule_holds_the_kernels_constants():
    import os
    import re
    src = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_01654_gb300",
                            "csrc", "mppi_iter.cuh")).read()
    const = {k: eval(v.replace("f", "").replace("CERT_CAP", "12.0"))
             for k, v in re.findall(r"constexpr float (CERT_\w+) = ([^;]+);", src)}
    assert const == {"CERT_CAP": CAP, "CERT_FAR": FAR, "CERT_LONG": LONG}
