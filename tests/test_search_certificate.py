"""The closest-point search's certificates and its ordering of near ties (no GPU).

The rollout kernel accepts the winner of a window of three segments (or vertices) when its computed
squared distance is within the winner's certificate, and orders two neighbours whose binary32 distances
nearly tie from the signs of two projections instead of in binary64.  Both rest on arguments about
geometry and rounding; here they are restated in numpy (the distances in binary32, operation by
operation, as the kernel takes them; the certificates in binary64, from the same formulas) and checked
on adversarial lanes and points: no accepted winner may differ from the brute-force minimum, and no
decided tie from the binary64 order.
"""
import numpy as np
import pytest

from test_search_bound import F, fma, lane, points_near, points_past_ends, seg_dist2, seg_records

CAP = 12.0


def smooth_lane(rng, n, spacing, bend, heading, origin):
    """A gently bending lane of near-equal segments: heading changes by up to `bend` rad a segment."""
    ang = heading + np.cumsum(bend * np.sin(np.arange(n - 1) * rng.uniform(0.01, 0.3)))
    ln = spacing * rng.uniform(0.98, 1.02, n - 1)
    w = np.zeros((n, 2))
    w[0] = origin + rng.uniform(-50.0, 50.0, 2)
    w[1:] = w[0] + np.cumsum(np.stack([ln * np.cos(ang), ln * np.sin(ang)], 1), 0)
    return (w[:, 0] - origin[0]).astype(F), (w[:, 1] - origin[1]).astype(F)


def unit(dx, dy):
    ln = np.hypot(dx, dy)
    return (dx / ln, dy / ln, ln) if ln > 0 else (0.0, 0.0, 0.0)


def cert_segments(x, y):
    """Certificates (distances) of the segments of a polyline, in binary64."""
    x, y = x.astype(np.float64), y.astype(np.float64)
    n = len(x) - 1
    out = np.zeros(n)
    for i in range(n):
        tx, ty, ln = unit(x[i + 1] - x[i], y[i + 1] - y[i])
        if ln == 0:
            continue
        lens = [ln]
        sp = sm = 1.0
        op = om = 0.0
        nxt = unit(x[i + 2] - x[i + 1], y[i + 2] - y[i + 1]) if i + 1 < n else None
        prv = unit(x[i - 1] - x[i], y[i - 1] - y[i]) if i > 0 else None
        lens += [v[2] for v in (nxt, prv) if v]
        lmin, lmax = min(lens), max(lens)
        if lmin == 0:
            continue
        r0 = 0.25 * lmin
        omega = np.sqrt(2.0 ** -19 * (1 + lmax / r0)) + 2.0 ** -20 * (CAP + lmax) / lmin + 2e-6
        if nxt and tx * nxt[0] + ty * nxt[1] > 0:
            c = tx * nxt[1] - ty * nxt[0]
            sp, op = min(abs(c) + omega, 1.0), -1.0 if c > 0 else 1.0
        if prv and tx * prv[0] + ty * prv[1] < 0:
            c = tx * prv[1] - ty * prv[0]
            sm, om = min(abs(c) + omega, 1.0), -1.0 if c > 0 else 1.0
        omega = min(omega, 1.0)
        gap = 2.2 * r0 + 2.0 ** -18 * lmax
        ax, ay = (x[:-1] - x[i]) * tx + (y[:-1] - y[i]) * ty, (y[:-1] - y[i]) * tx - (x[:-1] - x[i]) * ty
        bx, by = (x[1:] - x[i]) * tx + (y[1:] - y[i]) * ty, (y[1:] - y[i]) * tx - (x[1:] - x[i]) * ty
        fwd, bwd = np.minimum(ax, bx) - ln, -np.maximum(ax, bx)
        gx = np.maximum(np.maximum(fwd, bwd), 0.0)
        ahead = fwd > bwd
        s = np.where(gx > 0, np.where(ahead, sp, sm), max(sp, sm))
        o = np.where(ahead, op, om)
        yn = np.where(np.where(ahead, ax <= bx, ax >= bx), ay, by)
        ymax = np.maximum(abs(ay), abs(by))
        ymin = np.where(ay * by <= 0, 0.0, np.minimum(abs(ay), abs(by)))
        dxj = abs(bx - ax)
        lj = np.maximum(ln, dxj + abs(by - ay))
        c2, bl, qa = 2.0 ** -37 * lj * lj, 1.016 * 2.0 ** -19 * lj, 1.016 * 2.0 ** -18
        g2 = gx * gx + ymin * ymin
        n1, n2 = g2 - c2, gx * gx - c2
        nn = np.maximum(yn + gx * np.where(o >= 0, s, omega), -yn + gx * np.where(o <= 0, s, omega))
        b1, b2, a1 = ymax + gx * s + bl, np.maximum(nn, 0.0) + bl, s * s + qa
        with np.errstate(all="ignore"):
            r1 = n1 / (b1 + np.sqrt(b1 * b1 + a1 * np.maximum(n1, 0)))
            r2 = np.minimum(n2 / (b2 + np.sqrt(b2 * b2 + qa * np.maximum(n2, 0))),
                            gx * dxj / (s * dxj + abs(by - ay)))
        r = np.maximum(np.where(n1 > 0, r1, 0.0), np.where((n2 > 0) & (dxj > 0), r2, 0.0))
        r = np.where(g2 >= gap * gap, r, 0.0)
        r[max(i - 1, 0):i + 2] = CAP
        out[i] = 0.9 * min(CAP, r.min())
    return out


def cert_vertices(x, y):
    x, y = x.astype(np.float64), y.astype(np.float64)
    n = len(x)
    out = np.zeros(n)
    for i in range(n):
        wx, wy = x - x[i], y - y[i]
        w2 = wx * wx + wy * wy
        r = np.sqrt(w2) / 2.1
        for k in (i - 1, i + 1):                # the next vertex's side counts before the previous one's
            if not 0 <= k < n:
                continue
            tx, ty, ln = unit(x[k] - x[i], y[k] - y[i])
            if ln == 0:
                continue
            xs, ys = wx * tx + wy * ty, abs(wy * tx - wx * ty)
            num, qa = w2 - xs * ln, 1.016 * 2.0 ** -20 * (2 * xs / ln + 3)
            with np.errstate(all="ignore"):
                v = np.where(num > 0, num / (ys + np.sqrt(ys * ys + qa * np.maximum(num, 0))), 0.0)
            r = np.where(xs >= 0, v, r)
        r[max(i - 1, 0):i + 2] = CAP
        out[i] = 0.9 * min(CAP, r.min())
    return out


LANES = ["straight", "zigzag", "walk", "gentle", "bent", "dense"]


def make_lane(rng, kind, scale):
    origin = rng.uniform(-1.0, 1.0, 2) * scale
    if kind in ("straight", "zigzag", "walk"):
        return lane(rng, kind, 60, origin)
    spacing, bend = {"gentle": (0.5, 0.01), "bent": (0.5, 0.15), "dense": (0.1, 0.002)}[kind]
    x, y = smooth_lane(rng, 80, spacing, bend, rng.uniform(-np.pi, np.pi), np.zeros(2))
    return (x + F(origin[0])).astype(F), (y + F(origin[1])).astype(F)     # far from the frame's origin


def points(rng, x, y, m):
    a, b = points_near(rng, x, y, m), points_past_ends(rng, x, y, m // 4)
    return np.concatenate([a[0], b[0]]), np.concatenate([a[1], b[1]])


@pytest.mark.parametrize("kind", LANES)
@pytest.mark.parametrize("scale", [0.0, 3e2, 1e4])
def test_an_accepted_window_holds_the_closest_segment(kind, scale):
    rng = np.random.default_rng([LANES.index(kind), int(scale), 1])
    accepted = 0
    for _ in range(6):
        x, y = make_lane(rng, kind, scale)
        px, py = points(rng, x, y, 2000)
        ex, ey, sz, sw = seg_records(x, y)
        d = seg_dist2(px[:, None], py[:, None], x[None, :-1], y[None, :-1], ex, ey, sz, sw)
        first = d.argmin(1)                                     # ties to the lowest index
        pad = np.pad(d, ((0, 0), (1, 1)), constant_values=np.inf)
        wins = (d < pad[:, :-2]) & (d <= pad[:, 2:])            # against the lower and the upper neighbour
        ok = wins & (d <= ((cert_segments(x, y).astype(F)) ** 2)[None, :])
        k, i = np.nonzero(ok)
        assert (i == first[k]).all()
        accepted += len(np.unique(k))
    if kind in ("straight", "gentle", "dense"):                 # the lanes it is for: most points
        assert accepted > 6 * 1250 if kind != "straight" else accepted > 0


@pytest.mark.parametrize("kind", LANES)
@pytest.mark.parametrize("scale", [0.0, 3e2, 1e4])
def test_an_accepted_window_holds_the_closest_vertex(kind, scale):
    rng = np.random.default_rng([LANES.index(kind), int(scale), 2])
    for _ in range(6):
        x, y = make_lane(rng, kind, scale)
        px, py = points(rng, x, y, 2000)
        dx, dy = (px[:, None] - x[None, :]).astype(F), (py[:, None] - y[None, :]).astype(F)
        d = fma(dx, dx, (dy * dy).astype(F))
        pad = np.pad(d, ((0, 0), (1, 1)), constant_values=np.inf)
        ok = (d < pad[:, :-2]) & (d <= pad[:, 2:]) & (d <= ((cert_vertices(x, y).astype(F)) ** 2)[None, :])
        k, i = np.nonzero(ok)
        assert (i == d.argmin(1)[k]).all()


def dist2_f64(px, py, ax, ay, bx, by):
    """seg_dist2_f64: binary64 distance from binary32 inputs."""
    px, py, ax, ay, bx, by = (v.astype(np.float64) for v in (px, py, ax, ay, bx, by))
    ex, ey = bx - ax, by - ay
    l2 = ex * ex + ey * ey
    with np.errstate(all="ignore"):
        tau = np.where(l2 > 0, ((px - ax) * ex + (py - ay) * ey) / np.where(l2 > 0, l2, 1.0), 0.0)
    qx = np.where(tau <= 0, ax, np.where(tau >= 1, bx, ax + tau * ex))
    qy = np.where(tau <= 0, ay, np.where(tau >= 1, by, ay + tau * ey))
    return (px - qx) ** 2 + (py - qy) ** 2


@pytest.mark.parametrize("kind", LANES)
@pytest.mark.parametrize("scale", [0.0, 3e2, 1e4])
def test_ties_decided_by_projections_are_in_binary64_order(kind, scale):
    rng = np.random.default_rng([LANES.index(kind), int(scale), 3])
    decided = 0
    for _ in range(6):
        x, y = make_lane(rng, kind, scale)
        px, py = points(rng, x, y, 8000)
        ex, ey, sz, sw = seg_records(x, y)
        lo = rng.integers(0, len(x) - 2, len(px))
        # half of the points around the shared vertex, at distances and angles of near ties
        v = lo + 1
        at = rng.integers(0, 2, len(px)).astype(bool)
        off, ang = np.exp(rng.uniform(np.log(1e-4), np.log(10.0), len(px))), rng.uniform(-np.pi, np.pi, len(px))
        nrm = np.arctan2(ey[v], ex[v]) + rng.choice([-0.5, 0.5], len(px)) * np.pi
        ang = np.where(rng.random(len(px)) < 0.7, nrm + rng.normal(0, 1, len(px)) * 10.0 ** rng.uniform(-7, -1, len(px)),
                       ang)
        px = np.where(at, (x[v] + off * np.cos(ang)).astype(F), px)
        py = np.where(at, (y[v] + off * np.sin(ang)).astype(F), py)
        wx, wy = (px - x[v]).astype(F), (py - y[v]).astype(F)
        fl, fu = fma(wx, sz[lo], (wy * sw[lo]).astype(F)), fma(wx, sz[v], (wy * sw[v]).astype(F))
        k = fma(F(2.0 ** -17), (abs(wx) + abs(wy)).astype(F), F(1e-5))
        ml, mu = (k * (abs(sz[lo]) + abs(sw[lo])).astype(F)), (k * (abs(sz[v]) + abs(sw[v])).astype(F))
        dl = dist2_f64(px, py, x[lo], y[lo], x[v], y[v])
        du = dist2_f64(px, py, x[v], y[v], x[v + 1], y[v + 1])
        valid = (ml > 0) & (mu > 0)
        both, upper, lower = (valid & (fl >= ml) & (fu <= -mu), valid & (fl >= ml) & (fu >= mu),
                              valid & (fl <= -ml) & (fu <= -mu))
        assert (dl[both] == du[both]).all()
        assert (du[upper] < dl[upper]).all() and (dl[lower] < du[lower]).all()
        decided += int(both.sum() + upper.sum() + lower.sum())
    assert decided > 6 * 4000
