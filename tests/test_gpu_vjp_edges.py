"""The force VJP where its kernels have edges: group halves and remainders, few groups shared by several warps,
leaves larger than a tile, massless cells, coincident particles, unsoftened pairs; against the
oracle's VJP on the same tree.

Bounds, before any run: as the parity tests of the same quantity (test_gpu_adjoint.py): 1e-10 of the largest
component in FP64, 2e-4 in FP32.
"""
import numpy as np
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu


def _plummer(n):
    x, _, m = inputs.plummer(n, 51)
    return x, m


def _massless(n):
    """A third of the particles massless, whole cells of them among the rest, and a clump of coincident ones."""
    x, m = _plummer(n)
    m[x[0] > 0.4] = 0.0
    x[:, 10:60] = x[:, 10:11] + 0.0
    return x, m


CASES = [
    ("n1", lambda: _plummer(1), dict()),
    ("n2", lambda: _plummer(2), dict()),
    ("n17_g16", lambda: _plummer(17), dict(group_size=16, theta=0.0)),
    ("n33_g64", lambda: _plummer(33), dict(group_size=64, theta=0.0)),
    ("n47_g64", lambda: _plummer(47), dict(group_size=64, theta=1.0, leaf_cap=1)),
    ("n700_direct", lambda: _plummer(700), dict(theta=0.0, order=0)),
    ("massless", lambda: _massless(3001), dict(theta=0.8)),
    ("massless_leaf1", lambda: _massless(1500), dict(theta=1.0, leaf_cap=1, group_size=64)),
    ("unsoftened", lambda: _plummer(900), dict(eps=0.0, theta=0.9)),
]


@pytest.mark.parametrize("precision,tol", [("f64", 1e-10), ("f32", 2e-4)])
@pytest.mark.parametrize("name,gen,p", CASES, ids=[c[0] for c in CASES])
def test_vjp_edges(orc, name, gen, p, precision, tol):
    from paper_2412_01733_gb300 import treegb as tg
    dt = torch.float64 if precision == "f64" else torch.float32
    x, m = (t.to("cuda", dt).contiguous() for t in gen())
    n = x.shape[1]
    p = dict(dict(eps=0.05, theta=0.7, order=2, leaf_cap=8, group_size=32), **p)
    g = torch.Generator().manual_seed(2)
    ab = torch.randn((3, n), generator=g, dtype=torch.float64).to("cuda", dt)
    pb = torch.randn(n, generator=g, dtype=torch.float64).to("cuda", dt)
    f64 = lambda t: t.double().cpu().numpy()
    with tg.Workspace(n, precision=precision, **p) as ws:
        ws.build(x); ws.moments(x, m); ws.forces(lists_only=True)
        xb, mb = ws.forces_adjoint(ab, pb)
        assert ws.status() == 0
        kw = dict(eps=p["eps"], quad=p["order"] == 2)
        r = orc.tree_forces(f64(x), f64(m), theta=p["theta"], lcap=p["leaf_cap"], gs=p["group_size"], **kw)
        xo, mo = orc.tree_forces_vjp(r, f64(x), f64(m), f64(ab), f64(pb), **kw)
        # (the masses of massless particles: a massless cell passes its Mbar on as it stands, from its own centre)
        w = f64(m) != 0.0
        for a, b in ((f64(xb), xo), (f64(mb)[w], mo[w])):
            assert np.abs(a - b).max() <= tol * max(np.abs(b).max(), 1e-300)
