"""The planner's figure behind the choice between teams and lone warps: the
first launch's time on so many runners, in chunks (an entry: two, and its
chunks, both visits of a whole cell's task; a cut cell's top part runs after
the subtree that ends last).  Values worked out by hand."""
import numpy as np
import pytest

from paper_1810_12742_gb300 import hines as H


def _chain(n):
    return np.arange(-1, n - 1, dtype=np.int32)


def _plan(trees, **opts):
    return H.Plan([p.size for p in trees], np.concatenate(trees), host_only=True, even_cuts=True,
                  pack_compartments=1, **opts)


def test_equal_tasks_take_rounds():
    plan = _plan([_chain(10)] * 2000)
    assert plan.n_tasks == 2000
    assert plan.team_stretch(2000, 4000) == 1.0  # a team for every entry
    assert plan.team_stretch(1999, 4000) == 2.0  # two rounds against one
    assert plan.team_stretch(1216, 2432) == 2.0
    assert plan.team_stretch(700, 1400) == 1.5  # three against two
    assert plan.team_stretch(125, 250) == 2.0  # sixteen against eight
    assert plan.team_stretch(124, 250) == pytest.approx(250 / 124)  # far more entries: the fluid limit
    assert plan.team_stretch(1000, 1000) == 1.0


def test_a_long_task_hides_the_rounds():
    # 60 pieces of 16: 60 chunks, both visits, and two: 122; the others 4 each
    trees = [_chain(960)] + [_chain(10)] * 2000
    plan = _plan(trees)
    assert plan.team_stretch(1000, 2000) == 1.0
    # 101 teams: the long one, and 2000 others on 100: 20 rounds of 4, below 122
    assert plan.team_stretch(126, 252) == 1.0
    # 11 of 2001 entries are far fewer than a sixteenth
    assert plan.team_stretch(11, 22) == 2.0


def test_a_top_part_follows_its_cells_last_subtree():
    # a root piece of 16 with two arms of 2560: cut into a top part of one piece
    # and two subtrees of 160 chunks
    arm = 2560
    p = np.concatenate((_chain(16), [15], 16 + np.arange(arm - 1), [15], 16 + arm + np.arange(arm - 1))).astype(np.int32)
    plan = _plan([p])
    assert plan.n_tasks == 3
    # on one runner the subtrees one after the other, 2 (2 + 160), then the top part, 2 + 2; on two side by side
    assert plan.team_stretch(1, 2) == pytest.approx(328 / 166)
    assert plan.team_stretch(2, 4) == 1.0


def test_empty_and_arguments():
    assert H.Plan(np.zeros(0, np.int32), np.zeros(0, np.int32), host_only=True).team_stretch(8, 16) == 1.0
    plan = _plan([_chain(5)])
    L = H.lib()
    for teams, lone in ((0, 4), (4, 0)):
        with pytest.raises(H.HinesError):
            plan.team_stretch(teams, lone)
    assert L.hines_plan_team_stretch(None, 1, 2, None) == H.HINES_ERR_INVALID_ARG
