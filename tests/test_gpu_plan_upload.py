"""A plan is complete on the device when its creation returns: a first solve on
a stream that does not block on the legacy one (torch's streams, the host
pipeline's) gives what the same solve gives after a synchronisation."""
import numpy as np
import pytest

from tests.helpers import problem
from paper_1810_12742_gb300 import hines as H
from paper_1810_12742_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# one small cell (every copy below the driver's staging size), cells with top parts, many small cells
@pytest.mark.parametrize("sizes,times", [((37,), 1), ((20000, 900, 7000), 3), ((24, 310, 1, 77), 2000)])
@pytest.mark.parametrize("dtype", ["f64", "compensated"])
def test_first_solve_on_a_non_blocking_stream(sizes, times, dtype):
    import torch
    r = np.random.default_rng(31)
    trees = [I.random_chainy_tree(r, n, 0.05) for n in sizes]
    probs = [problem(p, r) for p in trees]
    t = torch.float64 if dtype == "f64" else torch.float32
    d, u, b = (torch.as_tensor(np.tile(np.concatenate([q[k] for q in probs]), times)).cuda().to(t) for k in "dub")
    ncomp, parent = np.tile([p.size for p in trees], times), np.tile(np.concatenate(trees), times)

    def solve(plan, x):
        return H.solve(plan, d, u, x) if dtype == "f64" else H.solve_compensated(plan, d, u, x)
    plan = H.Plan(ncomp, parent)
    torch.cuda.synchronize()
    want = solve(plan, b.clone())
    stream = torch.cuda.Stream()
    for _ in range(10):
        x = b.clone()
        torch.cuda.synchronize()
        first = H.Plan(ncomp, parent)
        with torch.cuda.stream(stream):
            got = solve(first, x)
        torch.cuda.synchronize()
        assert bool((got == want).all())
        assert first.status() == 0
