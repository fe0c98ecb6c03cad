"""The FP32 direct sum's packed kernel against a plain FP64 sum of Eq. 1.

Bound, before any run: a pair term carries at most about eight FP32 roundings
(5e-7 of it), 128 terms are summed plainly (at most 128 roundings of 6e-8 of
the sum of their magnitudes), the rest is compensated: 1e-5 of the sum of the
terms' magnitudes covers it.
"""
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu


def _reference(x, m, t, eps):
    """Accelerations, potentials and the sums of the terms' magnitudes (pairs with NaN or zero r^2 left out)."""
    x, m = x.double(), m.double()
    ok = (t >= 0) & (t < x.shape[1])
    p = x[:, t.clamp(0, x.shape[1] - 1)]
    d = x[:, None, :] - p[:, :, None]
    r2 = (d * d).sum(0) + eps * eps
    use = (r2 > 0) & (torch.arange(x.shape[1], device=x.device)[None] != t[:, None])
    ri = torch.where(use, r2.clamp(min=1e-300) ** -0.5, torch.zeros_like(r2))
    d = torch.where(use[None], d, torch.zeros_like(d))
    w = m * ri ** 3
    a, f = (w * d).sum(2), -(m * ri).sum(1)
    return torch.where(ok, a, a * float("nan")), torch.where(ok, f, f * float("nan")), (w * d).abs().sum(2), f.abs()


@pytest.mark.parametrize("eps", [0.01, 0.0])
@pytest.mark.parametrize("n,nt", [(1, 1), (2, 2), (127, 5), (129, 129), (3000, 255), (3001, 513), (40000, 1025)])
@pytest.mark.parametrize("nan", [False, True])
def test_direct_f32(n, nt, eps, nan):
    from paper_2412_01733_gb300 import treegb as tg
    x, _, m = (t.to("cuda", torch.float32).contiguous() for t in inputs.plummer(n, 4))
    if n > 200:
        x[:, 150] = x[:, 20]      # a coincident pair
    g = torch.Generator().manual_seed(n)
    t = torch.randint(0, n, (nt,), generator=g).cuda()  # repeated targets among them
    if nt > 4:
        t[3], t[4] = -1, n        # outside: NaN
    if nan and n > 200:
        x[1, 137] = float("nan")  # a source whose pairs have no distance
        t = torch.where(t == 137, torch.full_like(t, 20), t)
    with tg.Workspace(1, eps=eps) as ws:
        a, f = ws.direct(x, m, t)
    ar, fr, sa, sf = _reference(x, m, t, eps)
    assert torch.equal(a.isnan(), ar.isnan()) and torch.equal(f.isnan(), fr.isnan())
    assert ((a - ar).abs() <= 1e-5 * sa)[~ar.isnan()].all() and ((f - fr).abs() <= 1e-5 * sf)[~fr.isnan()].all()
