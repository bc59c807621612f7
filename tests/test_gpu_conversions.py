"""GPU test of the conversions between FP64 and double-float over the range of exponents
in which they change from integer steps to FP64 operations."""
import numpy as np
import pytest

from tests import gpu_helpers as gh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo", ["zero", "least", "small", "half"])
def test_round_trip_of_small_and_large_values(lo):
    """Y + X 0 gives back every y = hi + lo of two FP32 numbers: hi from 2^-97 to 2^97, powers
    of two among them, lo zero, subnormal (below 2^-126) or normal, of either sign."""
    dims = (4, 4, 4, 4)
    vh = 128
    s, _, _ = gh.make_solver(dims, 0.1, seed=85, max_rhs=2)
    e = np.arange(-97, 98)
    rng = np.random.default_rng(86)
    hi = np.ldexp(1.0 + rng.integers(0, 1 << 23, (8, e.size)) * 2.0 ** -23, e)
    hi[:2] = np.ldexp(1.0, e)
    q = {"zero": 0, "least": 1, "small": rng.integers(1, 1 << 10, hi.shape),
         "half": rng.integers(1 << 23, 1 << 24, hi.shape)}[lo]
    # lo in units of 2^(e - 52 + 2) (a power of two has half the room below), no finer than FP32
    unit = np.ldexp(1.0, np.maximum(e - 50, -149))
    y = hi + np.where(np.arange(8)[:, None] % 2, -1, 1) * q * unit
    h = y.astype(np.float32).astype(np.float64)
    assert np.array_equal(h + (y - h).astype(np.float32), y)  # two FP32 numbers hold it
    vals = np.concatenate([y.ravel(), -y.ravel()])
    for k in range(0, vals.size, 2 * 2 * vh * 3):
        flat = np.zeros(2 * 2 * vh * 3)
        part = vals[k:k + flat.size]
        flat[:part.size] = part
        block = flat.view(np.complex128).reshape(2, vh, 3)
        out = gh.to_np(s.block_caxpy(np.ones((2, vh, 3)), np.zeros((2, 2)), block))
        assert np.array_equal(out, block)
