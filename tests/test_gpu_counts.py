"""The counters a solve expects to find at 0 are 0 between calls, in every mode
and on both kinds of launch, and counters that are wrong when a call starts (as
calls on one plan that were not ordered find them) spoil that call only."""
import numpy as np
import pytest

from tests.helpers import problem
from paper_1810_12742_gb300 import hines as H
from paper_1810_12742_gb300 import inputs as I

pytestmark = pytest.mark.gpu

MODES = ["f64", "f32", "compensated", "refine", "cable step", "cable solve", "packed f64"]


def _plan(cells):
    """cells: "whole", 9000 tasks of one small cell (no cell cut, more tasks than any persistent grid has warps), or
    "cut", cells in parts: subtree tasks on teams (3 cells) or on lone warps (600)."""
    r = np.random.default_rng(41)
    if cells == "whole":
        trees, times = [I.random_chainy_tree(r, int(k), 0.2) for k in r.integers(1, 12, 9)], 1000
    else:
        bp = np.concatenate(([-1], np.zeros(10, np.int64)))
        trees, times = [I.compartments_from_branches(bp, r.integers(400, 600, 11))], 3 if cells == "cut, few" else 600
    probs = [problem(p, r) for p in trees]
    a = {k: np.tile(np.concatenate([q[k] for q in probs]), times) for k in ("d", "u", "b", "s")}
    plan = H.Plan(np.tile([p.size for p in trees], times), np.tile(np.concatenate(trees), times), pack_compartments=1)
    assert plan.n_tasks == {"whole": 9000, "cut, few": 33, "cut": 6600}[cells]
    return plan, a


def _run(plan, a, mode):
    import torch
    f64 = {k: torch.as_tensor(v).cuda() for k, v in a.items()}
    f = {k: v.float() for k, v in f64.items()}
    if mode == "f64":
        return H.solve(plan, f64["d"], f64["u"], f64["b"].clone())
    if mode == "f32":
        return H.solve(plan, f["d"], f["u"], f["b"].clone())
    if mode == "compensated":
        return H.solve_compensated(plan, f["d"], f["u"], f["b"])
    if mode == "refine":
        return H.solve_refine(plan, f["d"], f["u"], f["b"], steps=2)
    if mode == "packed f64":
        return H.unpack(plan, H.solve_packed(plan, H.pack(plan, f64["d"]), H.pack_coupling(plan, f64["u"]),
                                             H.pack(plan, f64["b"])))
    if mode == "cable solve":
        return H.cable_solve(plan, f64["s"], f64["s"], f64["u"], f64["b"].clone(), 0.025, 1)
    return H.cable_step(plan, f64["s"], f64["s"], f64["u"], f64["b"].clone(), 0.025, -65.0, 1)


@pytest.mark.parametrize("cells", ["whole", "cut, few", "cut"])
@pytest.mark.parametrize("mode", MODES)
def test_counts_are_zero_after_a_call_whatever_they_were_before(mode, cells):
    plan, a = _plan(cells)
    assert H.check_counts(plan) == 0
    want = _run(plan, a, mode)
    assert H.check_counts(plan, disturb=True) == 0
    _run(plan, a, mode)
    assert H.check_counts(plan) == 0
    plan.status()  # (a refinement of undefined numbers may warn)
    got = _run(plan, a, mode)
    assert bool((got == want).all())
    assert plan.status() == 0


def test_arguments():
    plan, _ = _plan("cut, few")
    L = H.lib()
    assert L.hines_check_counts(plan.handle, 0, None) == H.HINES_ERR_INVALID_ARG
    assert L.hines_check_counts(None, 0, None) == H.HINES_ERR_INVALID_ARG
