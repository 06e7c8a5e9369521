"""Lanes that meet themselves: no certificate settles the search on the meeting point (no GPU).

Where two branches of a lane share a point, neither segment (or vertex) there has a certificate (its
value is 0), and at distance zero the acceptance test must still fail: the window then hands over to the
whole search, which takes the lowest index.  The kernel's own comparison is read from its source.
"""
import os
import re

import numpy as np
import pytest

from test_gpu_search_crossings import LANES
from test_search_bound import F, fma, seg_dist2, seg_records
from test_search_certificate import cert_segments, cert_vertices

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_01654_gb300", "csrc",
                      "mppi_iter.cuh")
ACCEPT = re.findall(r"b2 (<=?) (?:c\.)?cert\[", open(SOURCE).read())


def accepted(d, cert):
    """Items that win against their neighbours within their certificates, as each place of the kernel
    asks it (the hinted window, the moved window, the window of vertices)."""
    assert len(ACCEPT) == 3
    pad = np.pad(d, ((0, 0), (1, 1)), constant_values=np.inf)
    lim = (cert.astype(F) ** 2)[None, :]
    within = np.logical_or.reduce([d <= lim if op == "<=" else d < lim for op in ACCEPT])
    return (d < pad[:, :-2]) & (d <= pad[:, 2:]) & within


def points():
    """The meeting point and points around it, all exact in binary32."""
    o = np.concatenate([[0.0], 2.0 ** -np.arange(1, 24), -(2.0 ** -np.arange(1, 24))])
    return np.concatenate([0.25 + o, 0.25 + 0 * o, 0.25 + o]).astype(F), np.concatenate([0 * o, o, o]).astype(F)


@pytest.mark.parametrize("name", list(LANES))
def test_no_segment_is_accepted_before_a_lower_one_as_close(name):
    x, y = (LANES[name]().T).astype(F)
    px, py = points()
    ex, ey, sz, sw = seg_records(x, y)
    d = seg_dist2(px[:, None], py[:, None], x[None, :-1], y[None, :-1], ex, ey, sz, sw)
    assert (d[0] == 0.0).sum() >= 2
    k, i = np.nonzero(accepted(d, cert_segments(x, y)))
    assert (i == d.argmin(1)[k]).all()


@pytest.mark.parametrize("name", list(LANES))
def test_no_vertex_is_accepted_before_a_lower_one_as_close(name):
    x, y = (LANES[name]().T).astype(F)
    px, py = points()
    dx, dy = (px[:, None] - x[None, :]).astype(F), (py[:, None] - y[None, :]).astype(F)
    d = fma(dx, dx, (dy * dy).astype(F))
    k, i = np.nonzero(accepted(d, cert_vertices(x, y)))
    assert (i == d.argmin(1)[k]).all()
