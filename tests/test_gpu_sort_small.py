"""The one-cluster sort of small systems equals the general passes bit for bit.

A workspace told to withhold the words of a sort tile that does not exist takes
the general passes (and loses nothing by it), so the same call on both is the
comparison: box, keys, permutation, and the forces and steps that follow.
"""
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu


def _plummer(n):
    return inputs.plummer(n, 21)[0]


def _clumps(n):
    """Coincident particles: runs of equal keys longer and shorter than the insertion's limit."""
    x = _plummer(n)
    x[:, : n // 4] = x[:, :1]
    x[:, n // 2: n // 2 + 20] = x[:, n // 2: n // 2 + 1]
    return x


def _tight(n, k, size):
    """k particles in a cell far below the 13 levels that are sorted first, the rest spread out."""
    x = _plummer(n)
    g = torch.Generator().manual_seed(n)
    x[:, torch.randperm(n, generator=g)[:k]] = 0.3 + size * torch.rand(3, k, generator=g, dtype=torch.float64)
    return x


# block and cluster edges, then the runs
CASES = [(f"plummer{n}", lambda n=n: _plummer(n)) for n in
         (1, 2, 31, 32, 33, 255, 1023, 1024, 1025, 2048, 2049, 4096, 4097, 8191, 8193, 30011, 65535, 65536)]
CASES += [("clumps", lambda: _clumps(5000)), ("clumps16k", lambda: _clumps(16384)),
          ("run20", lambda: _tight(3000, 20, 1e-5)), ("run32", lambda: _tight(9000, 32, 1e-6)),
          ("run33", lambda: _tight(9000, 33, 1e-6)), ("run5000", lambda: _tight(20000, 5000, 1e-4)),
          ("one_point", lambda: torch.ones(3, 700, dtype=torch.float64))]


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("name,gen", CASES, ids=[c[0] for c in CASES])
def test_small_sort_equals_general_passes(name, gen, precision):
    from paper_2412_01733_gb300 import treegb as tg
    dt = torch.float64 if precision == "f64" else torch.float32
    x = gen().to("cuda", dt).contiguous()
    n = x.shape[1]
    m = torch.full((n,), 1.0 / n, device="cuda", dtype=dt)
    with tg.Workspace(n, precision=precision) as small, tg.Workspace(n, precision=precision) as general:
        general.set_waits(withhold=(9, 1 << 20))
        states = []
        for ws in (small, general):
            xs, v = x.clone(), torch.zeros_like(x)
            a, f = ws.accel(xs, m)
            a0, f0 = a.clone(), f.clone()
            tree, lo = ws.export_tree(), ws.export_boxes()
            ws.leapfrog_step(xs, v, m, a, 0.01, phi=f)
            assert ws.status() == 0
            states.append((tree["keys"], tree["perm"], lo[0], lo[1], a0, f0, xs, v, a, f))
        for s, t in zip(*states):
            assert torch.equal(s, t)


def test_small_sort_nonfinite_axis():
    """A coordinate that is not finite raises the status bit and leaves the box to the finite ones, as before."""
    from paper_2412_01733_gb300 import treegb as tg
    x = _plummer(3000).to("cuda", torch.float32).contiguous()
    x[1, 7], x[2, :] = float("nan"), float("inf")
    with tg.Workspace(3000) as small, tg.Workspace(3000) as general:
        general.set_waits(withhold=(9, 1 << 20))
        for ws in (small, general):
            ws.build(x)
        assert small.status() == general.status() == tg.DEV_NONFINITE
        assert all(torch.equal(s, t) for s, t in zip(small.export_boxes(), general.export_boxes()))
