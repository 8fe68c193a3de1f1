"""A task runs by a team of two warps or by a lone warp, by a rule on the
number of work entries.  A cell's arithmetic does not depend on which: the
same cells in a small batch (teams) and repeated many times in a large one
(lone warps) give the same bits, in every mode, layout and factor placement."""
import numpy as np
import pytest

from paper_1810_12742_gb300 import hines as H
from paper_1810_12742_gb300 import inputs as I
from tests.helpers import problem

pytestmark = pytest.mark.gpu

REPEAT = 700  # cells x REPEAT entries: above every mode's bound for teams
DT, E = 0.025, -65.0


def _cells():
    r = np.random.default_rng(3)
    chain = np.arange(-1, 700, dtype=np.int32)
    bp, _ = I.grow_branch_tree(r, 60, 0.5, 0.2)
    return [chain, np.full(41, 0, np.int32) - (np.arange(41) == 0).astype(np.int32),
            I.compartments_from_branches(bp, r.integers(1, 33, 60)), I.random_recursive_tree(r, 300),
            I.random_chainy_tree(r, 500, 0.1), np.array([-1], np.int32),
            I.random_chainy_tree(r, 5200, 0.03)]  # the last is cut into a top part and subtrees


def _batch(times, **opts):
    import torch
    trees = _cells()
    r = np.random.default_rng(4)
    probs = [problem(p, r) for p in trees]
    extra = [dict(g=r.uniform(0.1, 1.0, p.size), V=r.uniform(-80, -50, p.size)) for p in trees]
    # (even cuts: aligned ones depend on where a cell starts in the batch)
    plan = H.Plan(np.tile([p.size for p in trees], times), np.tile(np.concatenate(trees), times),
                  pack_compartments=1, even_cuts=True, **opts)
    arrays = {k: np.concatenate([q[k] for q in probs]) for k in ("d", "u", "b", "s")}
    arrays.update({k: np.concatenate([q[k] for q in extra]) for k in ("g", "V")})
    return plan, {k: torch.as_tensor(np.tile(v, times)).cuda() for k, v in arrays.items()}


def _run(mode, layout, plan, a):
    packed = layout == "solver"
    f = {k: v.float() for k, v in a.items()}

    def put(v, coupling=False):
        return (H.pack_coupling if coupling else H.pack)(plan, v) if packed else v.clone()

    def out(v):
        return H.unpack(plan, v) if packed else v
    if mode in ("f64", "f32"):
        q = a if mode == "f64" else f
        return out((H.solve_packed if packed else H.solve)(plan, put(q["d"]), put(q["u"], True), put(q["b"])))
    if mode == "compensated":
        call = H.solve_compensated_packed if packed else H.solve_compensated
        return out(call(plan, put(f["d"]), put(f["u"], True), put(f["b"])))
    if mode == "refine":
        return H.solve_refine(plan, f["d"], f["u"], f["b"], steps=2)
    s, g, u, V = put(a["s"]), put(a["g"]), put(a["u"], True), put(a["V"])
    step = H.cable_step_packed if packed else H.cable_step
    if mode == "cable solve":
        return out((H.cable_solve_packed if packed else H.cable_solve)(plan, s, g, u, put(a["b"]), DT, 0))
    step(plan, s, g, u, V, DT, E, 1)
    if mode == "reuse":
        H.cable_step_reuse(plan, s, g, u, V, DT, E, 1, solver_layout=packed)
    else:
        step(plan, s, g, u, V, DT, E, 1)
    return out(V)


_MODES = [(m, lay, fac) for m in ("f64", "cable", "cable solve", "reuse") for lay in ("natural", "solver")
          for fac in (1, 2)] + [(m, lay, 0) for m in ("f32", "compensated") for lay in ("natural", "solver")]


@pytest.mark.parametrize("per_lane", [1, 2])
@pytest.mark.parametrize("mode,layout,factor", _MODES + [("refine", "natural", 0)])
def test_teams_and_lone_warps_agree_bit_for_bit(mode, layout, factor, per_lane):
    results = []
    for times in (1, REPEAT):
        plan, arrays = _batch(times, fp64_factor=factor, pieces_per_lane=per_lane)
        x = _run(mode, layout, plan, arrays)
        again = _run(mode, layout, plan, arrays)
        assert bool((x == again).all())
        assert plan.status() == 0
        results.append(x)
    n = results[0].numel()
    many = results[1].view(REPEAT, n)
    assert bool((many == results[0]).all())


@pytest.mark.parametrize("layout,factor", [("natural", 1), ("natural", 2), ("solver", 1), ("solver", 2)])
def test_a_step_that_reuses_the_factor_equals_a_full_step(layout, factor):
    for times in (1, REPEAT):
        plan, arrays = _batch(times, fp64_factor=factor)
        assert bool((_run("reuse", layout, plan, arrays) == _run("cable", layout, plan, arrays)).all())
