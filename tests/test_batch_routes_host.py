"""Which items of a batch run in the persistent launch and which as launches of their own (host
only): the workspace of the first holds schedule tables, that of the others only lanes."""
import pytest

import paper_1905_00444_gb300 as qfx
import rqc_inputs as ri


def runs_as_launches(plan):
    arr = (qfx.qfx.BatchItem * 1)(qfx.qfx.BatchItem(plan._h.value, 0, 1, 0, 1, 0))
    one, two = (int(qfx.qfx.lib.qfx_batch_workspace_bytes(arr, 1, slots)) for slots in (1, 2))
    return 2 * one - two < 1 << 20      # without the slots: the plan's tables, or also the schedule's


@pytest.mark.parametrize("grid,n_open,launches", [
    ((4, 5, 8), 18, False), ((4, 5, 8), 19, True),          # 256 and 512 tiles of 8 rows
    ((8, 3, 12), 18, False), ((8, 3, 12), 19, True),
    ((6, 6, 16), 13, False), ((6, 6, 16), 14, True),
    ((6, 6, 24), 8, False), ((6, 6, 24), 9, True),          # 512 and 1024 tiles of 64 rows
    ((4, 4, 16), 15, False), ((4, 4, 16), 16, True), ((7, 7, 24), 4, True)])
def test_large_steps_run_as_launches(grid, n_open, launches):
    rows, cols, depth = grid
    plan = qfx.Plan(qfx.Circuit(ri.rqc(rows, cols, depth, seed=1)), n_open=n_open)
    assert runs_as_launches(plan) == launches
    tree = qfx.Plan(qfx.Circuit(ri.rqc(rows, cols, depth, seed=1)), n_open=n_open, family="tree",
                    max_intermediate_bytes=1 << 30)
    assert runs_as_launches(tree)
