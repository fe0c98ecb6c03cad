"""The split walk of small systems equals the one-warp walk bit for bit.

A workspace made for more particles than the split walk serves keeps no tile
slots and takes the one-warp walk, so the same call on both is the comparison.
"""
import numpy as np
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu

BIG = 140000  # above the split walk's largest workspace in either precision


def _cusp(n, decades, seed=1):
    """Particles spread evenly in the logarithm of their radius: very many small walk groups."""
    rng = np.random.default_rng(seed)
    d = rng.normal(size=(3, n))
    x = 10.0 ** (-decades * rng.random(n)) * d / np.linalg.norm(d, axis=0)
    return torch.as_tensor(x), torch.full((n,), 1.0 / n, dtype=torch.float64)


def _clumps(n, seed=2):
    """Coincident particles in leaves larger than a tile, among a Plummer sphere."""
    x, _, m = inputs.plummer(n, seed)
    x[:, 50:117] = x[:, 50:51]
    x[:, 300:337] = x[:, 300:301]
    return x, m


def _plummer(n):
    x, _, m = inputs.plummer(n, 3)
    return x, m


CASES = [
    ("one", lambda: _plummer(1), dict()),
    ("two", lambda: _plummer(2), dict()),
    ("tile_edge_33", lambda: _plummer(33), dict(theta=0.0)),
    ("chunk_edge_513", lambda: _plummer(513), dict(theta=0.0)),          # 17 tiles of 32 sources: a second chunk
    ("direct_sum_3001", lambda: _plummer(3001), dict(theta=0.0, order=0)),
    ("clumps_g16", lambda: _clumps(2000), dict(group_size=16)),
    ("clumps_unsoftened", lambda: _clumps(2000), dict(eps=0.0)),
    ("plain_sums", lambda: _plummer(20011), dict(kahan=0)),
    ("monopole_chunks", lambda: _plummer(20011), dict(order=0, group_split=0)),
    ("g64", lambda: _plummer(20011), dict(group_size=64, leaf_cap=8, theta=0.5)),
    ("slots_run_out", lambda: _cusp(8000, 5), dict(group_size=16, group_split=1, theta=0.6, leaf_cap=1)),
]


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("name,gen,p", CASES, ids=[c[0] for c in CASES])
def test_split_walk_equals_one_warp_walk(name, gen, p, precision):
    from paper_2412_01733_gb300 import treegb as tg
    dt = torch.float64 if precision == "f64" else torch.float32
    x, m = (t.to("cuda", dt).contiguous() for t in gen())
    n = x.shape[1]
    p = dict(dict(eps=0.01, theta=0.7, precision=precision), **p)
    with tg.Workspace(n, **p) as split, tg.Workspace(BIG, **p) as plain:
        for _ in range(2):
            a, f = split.accel(x, m)
        a0, f0 = plain.accel(x, m)
        assert split.status() == 0 and plain.status() == 0
        assert torch.equal(a, a0) and torch.equal(f, f0)
        i, i0 = split.info(), plain.info()
        assert all(i[k] == i0[k] for k in ("pp_pairs", "pc_pairs", "max_stack", "n_groups"))
        # the same tree again after the parameters have changed which walk serves it
        split.set_params(theta=0.05)
        plain.set_params(theta=0.05)
        assert all(torch.equal(s, t) for s, t in zip(split.forces(), plain.forces()))


def test_split_walk_ensemble():
    from paper_2412_01733_gb300 import treegb as tg
    x, v, m, off = inputs.ensemble(5, 7, nmin=40, nmax=3000, device="cuda", dtype=torch.float32)
    x, m = x.contiguous(), m.contiguous()
    with tg.Workspace(x.shape[1], theta=0.6) as split, tg.Workspace(BIG, theta=0.6) as plain:
        for ws in (split, plain):
            ws.set_segments(off)
        assert all(torch.equal(s, t) for s, t in zip(split.accel(x, m), plain.accel(x, m)))
