"""The octree built straight from adjacent keys equals the level-by-level one.

A workspace for more than 65536 particles with a node array of its own size
builds level by level, so the same positions on both are the comparison: every
array of the tree and the walk groups, bit for bit.
"""
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu

BIG = 65537  # the smallest workspace that builds level by level (given a node array's size)


def _clumped(n):
    """Coincident particles (leaves at depth 21 holding more than leaf_cap) in a Plummer sphere."""
    x = inputs.plummer(n, 5)[0]
    x[:, n // 3: n // 3 + 40] = x[:, :1]
    x[:, n // 2: n // 2 + 17] = x[:, 1:2]
    return x


# sizes at the edges of a warp, a block, a block of several items, and of leaf_cap
SIZES = [1, 2, 8, 9, 16, 17, 31, 32, 33, 255, 256, 257, 1023, 131072, 131073, 262145, 524289, 1 << 20,
         (1 << 20) + 1, 3000001]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("leaf_cap", [1, 8, 16])
def test_flat_octree_equals_level_by_level(n, leaf_cap):
    from paper_2412_01733_gb300 import treegb as tg
    x = (_clumped(n) if n >= 255 else inputs.plummer(n, 5)[0]).to("cuda", torch.float32).contiguous()
    with tg.Workspace(n, leaf_cap=leaf_cap) as flat, tg.Workspace(max(n, BIG), leaf_cap=leaf_cap,
                                                                     node_cap=max(n, BIG) * 5) as level:
        for ws in (flat, level):
            ws.build(x)
        a, b = flat.export_tree(), level.export_tree()
        assert flat.status() == 0 and level.status() == 0
        assert a["info"]["level_offset"] == b["info"]["level_offset"]
        for k in ("keys", "perm", "level", "corner", "first", "count", "child", "nchild"):
            assert torch.equal(a[k], b[k]), k
        assert torch.equal(flat.export_groups(), level.export_groups())


@pytest.mark.parametrize("n,cap", [(20000, 3000), (20000, 3003), (3001, 9), (500, 1), (40, 40)])
def test_flat_octree_out_of_nodes_equals_level_by_level(n, cap):
    """A node array that is too small cuts the same tree in both forms."""
    from paper_2412_01733_gb300 import treegb as tg
    x, _, m = (t.to("cuda", torch.float32).contiguous() for t in inputs.plummer(n, 6))
    p = dict(theta=0.6, leaf_cap=2, node_cap=cap)
    with tg.Workspace(n, **p) as flat, tg.Workspace(BIG, **p) as level:
        out = [ws.accel(x, m) for ws in (flat, level)]
        st = [ws.status() for ws in (flat, level)]
        assert st[0] == st[1] == tg.DEV_NODES
        a, b = flat.export_tree(), level.export_tree()
        for k in ("keys", "perm", "level", "corner", "first", "count", "child", "nchild"):
            assert torch.equal(a[k], b[k]), k
        assert torch.equal(flat.export_groups(), level.export_groups())
        assert all(torch.equal(s, t) for s, t in zip(*out))


@pytest.mark.parametrize("sizes", [[1, 1], [1, 2, 17, 33, 700, 4101, 9000], [1] * 600 + [16] * 40 + [17, 3000],
                                   [255, 1, 256, 1, 2048, 16, 2032], [140000, 5, 140000]])
@pytest.mark.parametrize("leaf_cap,cap", [(16, 0), (1, 0), (4, 700)])
def test_flat_octree_of_systems(sizes, leaf_cap, cap):
    """Several systems (boundaries inside tiles, halos and leaves); cap: also when the node array is too small."""
    from paper_2412_01733_gb300 import treegb as tg
    off = [0]
    for k in sizes:
        off.append(off[-1] + k)
    n = off[-1]
    x = torch.cat([inputs.plummer(k, 70 + b % 7)[0] for b, k in enumerate(sizes)], 1).to("cuda", torch.float32).contiguous()
    if cap and len(sizes) >= cap:
        pytest.skip("more systems than nodes")
    with tg.Workspace(n, leaf_cap=leaf_cap, **(dict(node_cap=cap) if cap and n <= 65536 else {})) as flat, \
            tg.Workspace(max(n, BIG), leaf_cap=leaf_cap, node_cap=cap if cap and n <= 65536 else 5 * max(n, BIG)) as level:
        for ws in (flat, level):
            ws.set_segments(off)
            ws.build(x)
        a, b = flat.export_tree(), level.export_tree()
        assert flat.status() == level.status()
        for k in ("keys", "perm", "level", "corner", "first", "count", "child", "nchild"):
            assert torch.equal(a[k], b[k]), k
        assert torch.equal(flat.export_groups(), level.export_groups())
