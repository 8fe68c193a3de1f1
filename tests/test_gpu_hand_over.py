"""A large cell's top part goes to whoever finishes its last subtree, here a
lone warp (more work entries than any mode runs by teams): it has to see the
contributions the cell's other subtrees left from other multiprocessors.  All
copies of one cell hold the same numbers, so one missed contribution shows as
a copy that differs."""
import numpy as np
import pytest

import oracle
from tests.helpers import problem
from paper_1810_12742_gb300 import hines as H
from paper_1810_12742_gb300 import inputs as I

pytestmark = pytest.mark.gpu

COPIES, ARMS = 500, 12  # 6000 subtree tasks, 500 top parts


@pytest.mark.parametrize("per_lane", [1, 2])
@pytest.mark.parametrize("dtype", ["f64", "f32", "compensated"])
def test_top_parts_taken_over_by_lone_warps(dtype, per_lane):
    import torch
    r = np.random.default_rng(21)
    lens = np.concatenate(([400], r.integers(350, 500, ARMS)))  # (no subtree above 4096 compartments: one unit an arm)
    p = I.compartments_from_branches(np.concatenate(([-1], np.zeros(ARMS, np.int64))), lens)
    np_t = np.float64 if dtype == "f64" else np.float32
    q = {k: v.astype(np_t) for k, v in problem(p, r).items()}
    plan = H.Plan(np.full(COPIES, p.size), np.tile(p, COPIES), pack_compartments=1, even_cuts=True,
                  pieces_per_lane=per_lane)
    assert plan.n_tasks == COPIES * (ARMS + 1)
    d, u, b = (torch.as_tensor(np.tile(q[k], COPIES)).cuda() for k in ("d", "u", "b"))
    ref = oracle.solve_batch(np.array([p.size], np.int32), p, *(q[k].astype(np.float64) for k in ("d", "u", "b")))
    gate = {"f64": 1e-12, "f32": 1e-5, "compensated": 1e-10}[dtype]  # the solver's stated tolerances
    for _ in range(20):
        x = H.solve_compensated(plan, d, u, b) if dtype == "compensated" else H.solve(plan, d, u, b.clone())
        x = x.view(COPIES, p.size)
        assert bool((x == x[0]).all())
        assert np.abs(x[0].cpu().numpy() - ref).max() <= gate * np.abs(ref).max()
    assert plan.status() == 0
