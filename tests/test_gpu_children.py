"""Pieces with none, one, two, three and very many children, side by side in a
chunk, in tasks of teams (few cells) and of lone warps (many copies): every
mode against the oracle, every copy the same bits."""
import numpy as np
import pytest

import oracle
from paper_1810_12742_gb300 import hines as H

pytestmark = pytest.mark.gpu


def _cells():
    """Cells of up to 4096 compartments: whole tasks, so that all children of a piece are in its task."""
    star = np.zeros(700, np.int32)
    star[0] = -1
    r = np.random.default_rng(61)
    mixed = [-1]  # a chain whose compartments carry 0 to 6 leaves each
    tip = 0
    for k in range(150):
        for _ in range(int(r.integers(0, 7))):
            mixed.append(tip)
        mixed.append(tip)
        tip = len(mixed) - 1
    binary = np.array([-1] + [(i - 1) // 2 for i in range(1, 1023)], np.int32)
    return [star, np.array(mixed, np.int32), binary]


@pytest.mark.parametrize("per_lane", [1, 2])
@pytest.mark.parametrize("mode", ["f64", "f32", "compensated", "refine"])
@pytest.mark.parametrize("layout", ["natural", "solver"])
def test_any_number_of_children(layout, mode, per_lane):
    import torch
    if mode == "refine" and layout == "solver":
        pytest.skip("the refinement takes natural-layout arrays")
    t = torch.float64 if mode == "f64" else torch.float32
    gate = {"f64": 1e-12, "f32": 1e-5, "compensated": 1e-10, "refine": 1e-10}[mode]  # the solver's stated tolerances
    for p in _cells():
        r = np.random.default_rng(62)
        n = p.size
        # (a margin of 0.1 of the couplings, as the workloads' largest)
        a = r.uniform(0.5, 2.0, n)
        a[0] = 0.0
        sums = a + np.bincount(p[1:], weights=a[1:], minlength=n)
        d, u, b = (v.astype(np.float32).astype(np.float64) for v in (1.1 * sums, -a, r.uniform(-1, 1, n)))
        ref = oracle.solve_batch(np.array([n], np.int32), p, d, u, b)
        for copies in (3, 5000):  # 5000 tasks: above every mode's bound for teams
            plan = H.Plan(np.full(copies, n), np.tile(p, copies), pack_compartments=1, even_cuts=True,
                          pieces_per_lane=per_lane)
            dt, ut, bt = (torch.as_tensor(np.tile(v, copies)).cuda().to(t) for v in (d, u, b))
            if layout == "solver":
                q = H.pack(plan, dt), H.pack_coupling(plan, ut), H.pack(plan, bt)
                x = H.unpack(plan, H.solve_compensated_packed(plan, *q) if mode == "compensated"
                             else H.solve_packed(plan, *q))
            elif mode == "compensated":
                x = H.solve_compensated(plan, dt, ut, bt)
            elif mode == "refine":
                x = H.solve_refine(plan, dt, ut, bt, steps=2)
            else:
                x = H.solve(plan, dt, ut, bt)
            x = x.view(copies, n)
            assert bool((x == x[0]).all())
            assert np.abs(x[0].cpu().numpy() - ref).max() <= gate * np.abs(ref).max()
            assert plan.status() == 0
