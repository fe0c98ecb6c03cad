"""The autotuner's rows time the walk that a workspace created with the row's parameters runs.

In FP64 at 16384 particles the split walk takes a third of the one-warp walk's time or less, so a row that timed the
other one would be off by more than the factor two allowed here.
"""
import pytest
import torch

from paper_2412_01733_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base_group", [32, 16])
def test_rows_time_the_walk_of_their_parameters(base_group):
    from paper_2412_01733_gb300 import treegb as tg
    n, reps = 16384, 5
    x, _, m = (t.cuda().contiguous() for t in inputs.plummer(n, 33))
    p = dict(eps=0.01, theta=0.7, precision="f64")
    _, table = tg.autotune(x, m, reps=reps, max_err=None, group_size=base_group, **p)
    assert len(table) == 18
    for leaf_cap, group_size, stack, ms, _ in table:
        with tg.Workspace(n, leaf_cap=int(leaf_cap), group_size=int(group_size), stack_depth=int(stack), **p) as ws:
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            for r in range(reps + 1):
                if r == 1:
                    e[0].record()
                ws.build(x); ws.moments(x, m); ws.forces(want_phi=False)
            e[1].record()
            torch.cuda.synchronize()
        own = e[0].elapsed_time(e[1]) / reps
        assert ms <= 2.0 * own and own <= 2.0 * ms, (leaf_cap, group_size, stack, ms, own)
