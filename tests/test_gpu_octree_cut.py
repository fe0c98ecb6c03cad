"""A tree cut by its node array, built straight from adjacent keys, equals the level-by-level one, and takes the
whole chip as that one does.

A workspace for more than 65536 particles with a node array of its own size builds level by level; the default size of
the array is given there explicitly.  Tight pairs (triples) at leaf_cap 1 (2) need more nodes than the default holds.
"""
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu

FIELDS = ("keys", "perm", "level", "corner", "first", "count", "child", "nchild")


def _tight(n, k):
    """Particles in clumps of k, a cell or two of the finest level apart."""
    x = inputs.plummer(n, 21)[0]
    i = torch.arange(n)
    return x[:, i // k * k] + 3e-5 * (i % k)


def _default_cap(n, leaf_cap):
    return int(n * (8.0 / (leaf_cap + 1.0) + 0.25) + 4096.0)


def _equal(flat, level):
    assert flat.status() == level.status()
    a, b = flat.export_tree(), level.export_tree()
    assert a["info"]["level_offset"] == b["info"]["level_offset"]
    assert all(torch.equal(a[k], b[k]) for k in FIELDS)
    assert torch.equal(flat.export_groups(), level.export_groups())


@pytest.mark.parametrize("leaf_cap,need", [(1, 2361), (2, 1501), (8, 461)])
def test_every_small_node_array(leaf_cap, need):
    """Cuts at every place: numbers of slots left, levels of the cut, children of the last slots."""
    from paper_2412_01733_gb300 import treegb as tg
    n = 331
    x = _tight(n, leaf_cap + 1).to("cuda", torch.float32).contiguous()
    for cap in range(1, need + 30, need // 100):
        with tg.Workspace(n, leaf_cap=leaf_cap, node_cap=cap) as flat, \
                tg.Workspace(65537, leaf_cap=leaf_cap, node_cap=cap) as level:
            for ws in (flat, level):
                ws.build(x)
            _equal(flat, level)


@pytest.mark.parametrize("n,leaf_cap", [(70001, 1), (300007, 2), (1048577, 1), (3000001, 1), (3000001, 2)])
def test_default_node_array_too_small(n, leaf_cap):
    from paper_2412_01733_gb300 import treegb as tg
    x = _tight(n, leaf_cap + 1).to("cuda", torch.float32).contiguous()
    with tg.Workspace(n, leaf_cap=leaf_cap) as flat, tg.Workspace(n, leaf_cap=leaf_cap,
                                                                  node_cap=_default_cap(n, leaf_cap)) as level:
        ms = []
        for ws in (flat, level):
            best = float("inf")
            for _ in range(3):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                e[0].record(); ws.build(x); e[1].record()
                torch.cuda.synchronize()
                best = min(best, e[0].elapsed_time(e[1]))
            ms.append(best)
            assert ws.status(clear=False) == tg.DEV_NODES
        _equal(flat, level)
    # (one block building the whole tree takes tens to hundreds of times as long)
    assert ms[0] <= 3.0 * ms[1] + 0.2, ms


@pytest.mark.parametrize("leaf_cap,clump", [(1, 2), (16, 1)])  # cut, and whole
def test_systems_above_the_scan(leaf_cap, clump):
    """Several systems in the form that scans the blocks' counts, their boundaries in late blocks and at block edges."""
    from paper_2412_01733_gb300 import treegb as tg
    off = [0]
    for k in (1, 700000, 17, 2048, 16, 31, 400001, 2):
        off.append(off[-1] + k)
    n = off[-1]
    x = _tight(n, clump).to("cuda", torch.float32).contiguous()
    with tg.Workspace(n, leaf_cap=leaf_cap) as flat, tg.Workspace(n, leaf_cap=leaf_cap,
                                                                  node_cap=_default_cap(n, leaf_cap)) as level:
        for ws in (flat, level):
            ws.set_segments(off)
            ws.build(x)
        assert flat.status(clear=False) == (tg.DEV_NODES if clump > 1 else 0)
        _equal(flat, level)
