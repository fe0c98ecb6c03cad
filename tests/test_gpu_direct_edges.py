"""The FP32 direct sum where the left-out pair alone would spoil the sums: a target's own pair at an eps whose eps^-2
is past the FP32 range, and a coincident source of infinite mass at eps = 0 (a pair without a distance contributes
nothing); against a plain FP64 sum of Eq. 1.

Bound, before any run: as the packed kernel's test (test_gpu_direct.py), 1e-5 of the sum of the terms' magnitudes.
"""
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu


def _check(x, m, t, eps, use):
    from paper_2412_01733_gb300 import treegb as tg
    with tg.Workspace(1, eps=eps) as ws:
        a, f = ws.direct(x, m, t)
    xd, md = x.double(), m.double()
    d = xd[:, None, :] - xd[:, t, None]
    ri = torch.where(use, ((d * d).sum(0) + eps * eps).clamp(min=1e-300) ** -0.5, 0.0)
    md = torch.where(use, md[None], 0.0)
    w = md * ri ** 3
    ar, fr, sa = (w * d).sum(2), -(md * ri).sum(1), (w * d).abs().sum(2)
    assert ((a - ar).abs() <= 1e-5 * sa).all() and ((f - fr).abs() <= 1e-5 * fr.abs()).all()


@pytest.mark.parametrize("n,nt", [(2, 2), (129, 129), (3000, 255), (40000, 1025)])
@pytest.mark.parametrize("eps", [1e-19, 5e-20, 1e-21, 5e-23])
def test_direct_own_pair_at_tiny_eps(n, nt, eps):
    x, _, m = (t.to("cuda", torch.float32).contiguous() for t in inputs.plummer(n, 8))
    t = torch.randint(0, n, (nt,), generator=torch.Generator().manual_seed(n)).cuda()
    _check(x, m, t, eps, torch.arange(n, device="cuda")[None] != t[:, None])


def test_direct_coincident_infinite_mass():
    n = 700
    x, _, m = (t.to("cuda", torch.float32).contiguous() for t in inputs.plummer(n, 9))
    x[:, 300] = x[:, 20]
    m[300] = float("inf")
    t = torch.tensor([20], device="cuda")
    j = torch.arange(n, device="cuda")[None]
    _check(x, m, t, 0.0, (j != 20) & (j != 300))
