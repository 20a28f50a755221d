"""The binary64 pivots are divided by with correct rounding: the selected
inverse of a diagonal matrix is 1 / q in every bit (all products with zeros
leave the reciprocal as it is), over the normal exponents and random
mantissas, values next to powers of two among them."""
import numpy as np
import pytest

from tests.test_gpu_parity import q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("low,high", [(-1, 1), (-60, 60), (-1020, -995), (990, 1020), (-1020, 1020)])
def test_inverse_of_a_diagonal_matrix(q, low, high):
    n_s, n_t = 320, 12
    rng = np.random.default_rng(high - low)
    mant = rng.uniform(1.0, 2.0, (n_t, n_s))
    near = rng.random((n_t, n_s)) < 0.2
    mant[near] = 1.0 + rng.integers(-3, 4, int(near.sum())) * 2.0 ** -52
    A = np.ldexp(mant, rng.integers(low, high, (n_t, n_s)))
    ptr = np.arange(n_s + 1, dtype=np.int32)
    ctx = q.qsel_create_bt(n_s, n_t, ptr, ptr[:-1].copy(), A, np.zeros((n_t - 1, n_s)), precision=q.QSEL_FP64,
                           n_parts=1, overlap=0, n_samples=2)
    assert np.array_equal(ctx.diag_inv(), (1.0 / A).reshape(-1))
