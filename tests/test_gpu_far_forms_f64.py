"""The FP64 walk's two far-cell forms agree.

Positions (and eps) scaled by a power of two scale every force exactly; scaled
until the tree's cube has side 2^201, the r^-5 form is not taken, while r^-5
(at least 2^-1009 there) still is a normal number in the full form, so the two
runs take one form each.  Bound: both forms sum the same few thousand terms
with about forty roundings of 1.1e-16 each; 1e-13 of the largest component
covers it.
"""
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [(3001, dict()), (3001, dict(eps=0.0)), (20011, dict(group_size=64, theta=0.9)),
                                 (140001, dict(theta=1.0))])  # the last one is walked by one warp per group
def test_far_cell_forms_agree_f64(n, p):
    from paper_2412_01733_gb300 import treegb as tg
    x, _, m = (t.cuda().contiguous() for t in inputs.plummer(n, 61))
    p = dict(dict(eps=0.01, theta=0.7, precision="f64"), **p)
    with tg.Workspace(n, **p) as ws:
        a, f = ws.accel(x, m)
        assert ws.status() == 0
        s = 201 - int(ws.export_boxes()[1][0])
    with tg.Workspace(n, **dict(p, eps=p["eps"] * 2.0 ** s)) as ws:
        a2, f2 = ws.accel((x * 2.0 ** s).contiguous(), m)
        assert ws.status() == 0 and int(ws.export_boxes()[1][0]) == 201
    for u, v in ((a, a2 * 2.0 ** (2 * s)), (f, f2 * 2.0 ** s)):
        assert (u - v).abs().max() <= 1e-13 * u.abs().max()
