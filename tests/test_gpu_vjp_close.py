"""The force VJP where a power of 1/r of a pair at zero or tiny distance leaves the FP32 range: small softenings, and
neighbours closer than any far cell; against the oracle's VJP on the same tree.

The tiles of the lists are seldom full, and neither are the groups, so every case has lanes without a source and
places without a target.  Bounds, before any run: as the parity tests of the same quantity (test_gpu_adjoint.py),
1e-10 of the largest component in FP64, 2e-4 in FP32.
"""
import numpy as np
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu


def _pairs(x):
    """Every second particle 1e-6 beside its neighbour."""
    x = x.clone()
    n = x.shape[1] // 2 * 2
    x[:, 1:n:2] = x[:, 0:n:2] + 1e-6
    return x


@pytest.mark.parametrize("precision,tol", [("f64", 1e-10), ("f32", 2e-4)])
@pytest.mark.parametrize("order", [0, 2])
@pytest.mark.parametrize("eps,close,group_size", [(1e-6, False, 32), (1e-9, False, 64), (1e-15, False, 16),
                                                  (1e-15, False, 64), (0.0, True, 32), (3e-6, True, 64)])
def test_vjp_of_close_pairs(orc, eps, close, group_size, order, precision, tol):
    from paper_2412_01733_gb300 import treegb as tg
    dt = torch.float64 if precision == "f64" else torch.float32
    n = 1501
    x, _, m = inputs.plummer(n, 53)
    x, m = (_pairs(x) if close else x).to("cuda", dt).contiguous(), m.to("cuda", dt).contiguous()
    g = torch.Generator().manual_seed(4)
    ab = torch.randn((3, n), generator=g, dtype=torch.float64).to("cuda", dt)
    pb = torch.randn(n, generator=g, dtype=torch.float64).to("cuda", dt)
    f64 = lambda t: t.double().cpu().numpy()
    with tg.Workspace(n, precision=precision, eps=eps, theta=0.9, order=order, leaf_cap=8, group_size=group_size) as ws:
        ws.build(x); ws.moments(x, m); ws.forces(lists_only=True)
        xb, mb = ws.forces_adjoint(ab, pb)
        assert ws.status() == 0
    kw = dict(eps=eps, quad=order == 2)
    r = orc.tree_forces(f64(x), f64(m), theta=0.9, lcap=8, gs=group_size, **kw)
    xo, mo = orc.tree_forces_vjp(r, f64(x), f64(m), f64(ab), f64(pb), **kw)
    assert np.isfinite(xo).all() and np.isfinite(mo).all()
    for a, b in ((f64(xb), xo), (f64(mb), mo)):
        assert np.abs(a - b).max() <= tol * np.abs(b).max()
