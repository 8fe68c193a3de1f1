"""The FP64 pivot reciprocal through the public solve: a batch of
one-compartment cells has x = b / d with b = 1, so x is the kernel's
reciprocal of d itself."""
import numpy as np
import pytest

from paper_1810_12742_gb300 import hines as H

pytestmark = pytest.mark.gpu


def _reciprocals(d):
    import torch
    n = d.size
    plan = H.Plan(np.ones(n, np.int32), np.full(n, -1, np.int32))
    x = torch.ones(n, dtype=torch.float64, device="cuda")
    return H.solve(plan, torch.as_tensor(d).cuda(), torch.zeros_like(x), x).cpu().numpy()


# mantissas at the cuts of the three-part split (24 + 24 + 5 bits), both ends of the binade, and random
_MANTISSAS = {
    "random": lambda r, n: r.integers(0, 1 << 52, n),
    "low word only": lambda r, n: r.integers(0, 1 << 29, n),
    "top 24 bits": lambda r, n: r.integers(0, 1 << 23, n) << 29,
    "last 5 bits": lambda r, n: r.integers(0, 32, n),
    "just below 2": lambda r, n: (1 << 52) - 1 - r.integers(0, 1 << 30, n),
    "middle word full": lambda r, n: (r.integers(0, 1 << 23, n) << 29) | ((1 << 29) - 1),
}


@pytest.mark.parametrize("kind", list(_MANTISSAS))
def test_reciprocal_within_one_unit_of_the_last_place(kind):
    """Below 0.501 units of the last place, so next to the correctly rounded quotient at most, for every exponent
    whose reciprocal is normal, both signs."""
    r = np.random.default_rng(5)
    n = 2045 * 8
    m = _MANTISSAS[kind](r, n).astype(np.uint64)
    e = np.tile(np.arange(1, 2046, dtype=np.uint64), 8)
    e[m == 0] = np.minimum(e[m == 0], 2044)
    e = np.where(e == 2045, 1, e).astype(np.uint64)  # exponent 2045: 1/d is subnormal
    sign = r.integers(0, 2, n).astype(np.uint64)
    d = ((sign << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)
    got, want = _reciprocals(d).view(np.int64), (1.0 / d).view(np.int64)
    assert np.abs(got - want).max() <= 1


def test_reciprocal_outside_the_normal_range_is_what_the_fp64_form_gives():
    """Zero, subnormal, infinite and NaN pivots give no number, a reciprocal below the normal range is flushed."""
    bad = np.array([0.0, -0.0, 5e-324, 1e-310, np.inf, -np.inf, np.nan])
    assert np.isnan(_reciprocals(bad)).all()
    assert (_reciprocals(np.array([1.7976931348623157e308, -1e308])) == 0.0).all()
