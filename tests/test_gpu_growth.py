"""The refinement's growth check: a warp for a cell of few pieces, the block for
one of many, one to eight cells to a block.  A batch of well-conditioned cells
raises nothing; one cell whose corrections grow raises the warning wherever it
stands and whatever its size."""
import functools

import numpy as np
import pytest

from paper_1810_12742_gb300 import hines as H

pytestmark = pytest.mark.gpu

BLOCKS = 8 * 152  # blocks of the check at a time on this part


def _star(pieces):
    """A root with pieces - 1 single-compartment children: `pieces` pieces."""
    p = np.zeros(pieces, np.int32)
    p[0] = -1
    return p


def _good(pieces):
    u = np.full(pieces, -1.0, np.float32)
    d = np.full(pieces, 2.0, np.float32)
    d[0] = 2.0 * pieces
    return d, u


@functools.cache
def _growing(pieces):
    """A star whose root pivot p = d_0 - sum 1/d_i cancels so far that FP32's rounding leaves another number q: the
    factor's correction is p/q times the right one, and each step multiplies the error by 1 - p/q.  d_0 is searched
    among the FP32 numbers around the sum for the largest factor (q from FP32 solves of the unit right-hand side)."""
    import torch
    r = np.random.default_rng(72)
    d, u = np.float32(r.uniform(2.0, 3.0, pieces)), np.full(pieces, -1.0, np.float32)
    tail = float(np.sum(1.0 / np.float64(d[1:])))
    tries = np.float32(tail) + np.arange(-60, 61, dtype=np.float32) * np.spacing(np.float32(tail))
    dd = np.tile(d, tries.size)
    dd[::pieces] = tries
    plan = H.Plan(np.full(tries.size, pieces), np.tile(_star(pieces), tries.size))
    b = torch.zeros(dd.size, device="cuda")
    b[::pieces] = 1.0
    x = H.solve(plan, torch.as_tensor(dd).cuda(), torch.as_tensor(np.tile(u, tries.size)).cuda(), b)
    factor = np.abs(1.0 - (np.float64(tries) - tail) * x[::pieces].cpu().numpy().astype(np.float64))
    factor[~np.isfinite(factor) | (factor > 1e3)] = 0.0
    assert factor.max() > 2.0
    d[0] = tries[int(np.argmax(factor))]
    return d, u


# pieces of a cell around the line between a warp and a block (256), and a large one
@pytest.mark.parametrize("pieces", [60, 255, 256, 257, 258, 3000])
@pytest.mark.parametrize("cells", [1, 7, BLOCKS, BLOCKS + 1, 3 * BLOCKS + 5, 8 * BLOCKS + 3])
def test_the_largest_correction_of_every_cell_is_seen(pieces, cells):
    import torch
    small = 3
    for at in sorted({0, cells // 2, cells - 1}):  # among small cells, at the front, in the middle and at the end
        ncomp = np.full(cells, small)
        ncomp[at] = pieces
        parent = np.concatenate((np.tile(_star(small), at), _star(pieces), np.tile(_star(small), cells - 1 - at)))
        plan = H.Plan(ncomp, parent)
        b = torch.as_tensor(np.random.default_rng(71).uniform(-1, 1, parent.size)).cuda().float()
        for make, status in ((_good, 0), (_growing, H.HINES_WARN_REFINE), (_good, 0)):
            d, u = (torch.as_tensor(np.concatenate((np.tile(s, at), v, np.tile(s, cells - 1 - at)))).cuda()
                    for s, v in zip(_good(small), make(pieces)))
            H.solve_refine(plan, d, u, b, steps=2)  # (the second correction against the first)
            assert plan.status() == status
