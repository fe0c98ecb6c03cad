"""The moments' three forms (climbing from unsorted or sorted leaves, level by
level) give the same bits: the form follows the number of particles of the
build, so a system's moments are compared alone and beside a second system
that takes the build past each line.
"""
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu

FIELDS = ("M", "R", "Q")


def _system(n):
    x, _, m = inputs.plummer(n, 9)
    if n > 500:
        x[:, 100:160] = x[:, 100:101]   # a leaf of 60 at depth 21
        m[200:400] = 0.0                # massless cells
    return x, m


def _moments(ws, n):
    """Moments of the nodes of the first n particles, in breadth-first order."""
    t = ws.export_tree()
    mine = t["first"].long() < n
    M, R, Q = ws.export_moments()
    return M[mine], R[:, mine], Q[:, mine], t["level"][mine]


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("n", [1, 16, 17, 3001])
@pytest.mark.parametrize("other", [1 << 17, 1 << 20])
def test_moments_forms_agree(n, other, precision):
    from paper_2412_01733_gb300 import treegb as tg
    dt = torch.float64 if precision == "f64" else torch.float32
    x, m = _system(n)
    y, _, k = inputs.plummer(other, 10)
    xe, me = torch.cat((x, y), 1).to("cuda", dt).contiguous(), torch.cat((m, k)).to("cuda", dt).contiguous()
    x, m = x.to("cuda", dt).contiguous(), m.to("cuda", dt).contiguous()
    with tg.Workspace(n, precision=precision) as alone, tg.Workspace(n + other, precision=precision) as both:
        both.set_segments([0, n, n + other])
        for ws, a, b in ((alone, x, m), (both, xe, me)):
            for _ in range(2):  # a second pass finds the arrival counters clear
                ws.build(a)
                ws.moments(a, b)
        got, want = _moments(alone, n), _moments(both, n)
        assert all(torch.equal(s, t) for s, t in zip(got, want))
