"""A hines_cable_solve leaves the same factor as a full cable step: a step that
re-uses it afterwards equals a full step bit for bit, on a fresh plan (nothing
else has written the workspace) and after a step with another matrix."""
import numpy as np
import pytest

from tests.helpers import problem
from paper_1810_12742_gb300 import hines as H
from paper_1810_12742_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DT, E = 0.025, -65.0


@pytest.mark.parametrize("per_lane", [1, 2])
@pytest.mark.parametrize("layout", ["natural", "solver"])
@pytest.mark.parametrize("fp64_factor", [1, 2])
@pytest.mark.parametrize("theta", [0, 1])
def test_reuse_after_a_cable_solve(theta, fp64_factor, layout, per_lane):
    import torch
    r = np.random.default_rng(51)
    trees = [I.random_chainy_tree(r, n, 0.1) for n in (1, 17, 640, 5200)]  # the last is cut into parts
    a = {k: torch.as_tensor(np.concatenate([problem(p, np.random.default_rng(i))[k] for i, p in enumerate(trees)])).cuda()
         for k in ("s", "u", "b")}
    n = a["s"].numel()
    g, V0 = (torch.as_tensor(r.uniform(lo, hi, n)).cuda() for lo, hi in ((0.1, 1.0), (-80.0, -50.0)))
    packed = layout == "solver"

    def plan_and_arrays():
        plan = H.Plan([p.size for p in trees], np.concatenate(trees), fp64_factor=fp64_factor, pieces_per_lane=per_lane)
        if not packed:
            return plan, (a["s"], g, a["u"]), a["b"].clone(), V0.clone()
        return plan, (H.pack(plan, a["s"]), H.pack(plan, g), H.pack_coupling(plan, a["u"])), H.pack(plan, a["b"]), \
            H.pack(plan, V0)
    step, solve = (H.cable_step_packed, H.cable_solve_packed) if packed else (H.cable_step, H.cable_solve)
    plan, m, _, want = plan_and_arrays()
    step(plan, *m, want, DT, E, theta)
    for other_first in (False, True):
        plan, m, y, V = plan_and_arrays()
        if other_first:
            step(plan, *m, V.clone(), 3 * DT, E, theta)
        solve(plan, *m, y, DT, theta)
        H.cable_step_reuse(plan, *m, V, DT, E, theta, solver_layout=packed)
        got, ref = (H.unpack(plan, V), H.unpack(plan, want)) if packed else (V, want)
        assert bool((got == ref).all())
        assert plan.status() == 0
