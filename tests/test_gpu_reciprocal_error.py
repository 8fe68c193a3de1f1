"""The FP64 pivot reciprocal's error in units of the last place, exactly (whole
numbers), below 0.501: half a unit for the last rounding, and less than a
thousandth for what the form leaves out.  With |e| = |1 - m r| below 2^-22 (2^-23
from the reciprocal of the upper 24 bits, 2^-23 from the lower 29): e^3 is below
2^-66, 2^-13 of a unit (2^-53); the FP32 roundings of e's parts, of the product's
remainder (below 512 units) and of its correction are below 2^-15 of a unit each."""
import numpy as np
import pytest

from tests.test_gpu_reciprocal import _MANTISSAS, _reciprocals

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", list(_MANTISSAS))
def test_reciprocal_error_below_501_thousandths_of_a_unit(kind):
    r = np.random.default_rng(91)
    n = 40000
    m = _MANTISSAS[kind](r, n).astype(np.uint64)
    e = r.integers(1, 2045, n).astype(np.uint64)
    d = ((r.integers(0, 2, n).astype(np.uint64) << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)
    x = _reciprocals(d)
    assert (np.sign(x) == np.sign(d)).all()
    worst = 0.0
    for a, b in zip(np.abs(d), np.abs(x)):
        (fa, ea), (fb, eb) = np.frexp(a), np.frexp(b)
        ma, mb = int(fa * 2.0 ** 53), int(fb * 2.0 ** 53)  # a = ma 2^(ea - 53), b = mb 2^(eb - 53)
        # (b - 1/a) / 2^(eb - 53) = (ma mb - 2^(106 - ea - eb)) / ma
        worst = max(worst, abs(ma * mb - (1 << int(106 - ea - eb))) / ma)
    assert worst < 0.501
