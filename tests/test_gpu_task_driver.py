"""The task driver over the shapes of a launch: more entries than warps (the
work counter is used and restored), one entry per warp, tasks of one chunk up
to several windows of the chunk table, and cells whose top part is handed over
(their pending counts restored), each call repeated on one plan."""
import numpy as np
import pytest

import oracle
from tests.helpers import problem, relabel
from paper_1810_12742_gb300 import hines as H
from paper_1810_12742_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _chain(n):
    return np.arange(-1, n - 1, dtype=np.int32)


def _star_of_chains(arms, length):
    bp = np.concatenate(([-1], np.zeros(arms, np.int64)))
    return I.compartments_from_branches(bp, np.full(arms + 1, length))


_BATCHES = {
    # 9000 tasks of one small cell each: more than any persistent grid has warps
    "more tasks than warps": (lambda r: [I.random_chainy_tree(r, int(k), 0.2) for k in r.integers(1, 12, 9000)],
                              dict(pack_compartments=1)),
    "one cell": (lambda r: [I.random_chainy_tree(r, 37, 0.2)], {}),
    # 31 to 34 and 255 chunks of one piece: the chunk table's window edges
    "chains at the window edges": (lambda r: [_chain(16 * k) for k in (31, 32, 33, 34, 62, 63, 64, 255)],
                                   dict(pack_compartments=1)),
    # top parts: cells above 4096 compartments, wide and deep
    "handed-over top parts": (lambda r: [_star_of_chains(40, 300), _chain(9000), I.random_chainy_tree(r, 20000, 0.02)],
                              {}),
}


@pytest.mark.parametrize("name", list(_BATCHES))
@pytest.mark.parametrize("dtype", ["f64", "f32", "compensated"])
def test_repeated_calls_on_one_plan(name, dtype):
    import torch
    make, opts = _BATCHES[name]
    rng = np.random.default_rng(11)
    trees = make(rng)
    if name == "one cell":
        trees = [relabel(trees[0], rng)[0]]
    probs = [problem(p, rng) for p in trees]
    ncomp = np.array([p.size for p in trees], np.int32)
    parent = np.concatenate(trees)
    np_t = np.float64 if dtype == "f64" else np.float32
    d, u, b = (np.concatenate([q[k] for q in probs]).astype(np_t) for k in ("d", "u", "b"))
    plan = H.Plan(ncomp, parent, **opts)
    dt, ut, bt = (torch.as_tensor(v).cuda() for v in (d, u, b))
    got = []
    for _ in range(3):
        if dtype == "compensated":
            got.append(H.solve_compensated(plan, dt, ut, bt).cpu().numpy())
        else:
            got.append(H.solve(plan, dt, ut, bt.clone()).cpu().numpy())
    assert plan.status() == 0
    assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
    ref = oracle.solve_batch(ncomp, parent, *(v.astype(np.float64) for v in (d, u, b)))
    gate = {"f64": 1e-12, "f32": 1e-5, "compensated": 1e-10}[dtype]  # the solver's stated tolerances
    lo = 0
    for n in ncomp:
        x, y = got[0][lo:lo + n], ref[lo:lo + n]
        assert np.abs(x - y).max() <= gate * np.abs(y).max()
        lo += n
