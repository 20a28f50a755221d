"""The logarithms of the control-variate features, bit for bit: the float of
the logarithm of the same binary64 entries (long double here; where that and
the binary64 logarithm round to different floats, either).  Diagonal blocks
and couplings are given values: over the exponents, next to 1, sqrt(1/2),
sqrt(2) and powers of two, subnormal ones, and below the 1e-30 that couplings
are floored at."""
import numpy as np
import pytest

from tests.test_gpu_parity import q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

N_S, N_T = 2048, 96


def _values(rng, kind, shape):
    n = int(np.prod(shape))
    if kind == "exponents":
        v = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-1020, 1021, n))
    elif kind == "near_one":
        v = 1.0 + rng.choice([-1.0, 1.0], n) * 2.0 ** rng.uniform(-52.0, -1.0, n)
    elif kind == "ordinary":
        v = np.exp(rng.uniform(-12.0, 12.0, n))
    else:
        # a few units in the last place around the points where the method changes
        at = np.concatenate([np.sqrt([0.5, 2.0]), 2.0 ** np.arange(-40, 41), [2.0 ** -1022, 2.0 ** 1023]])
        v = rng.choice(at, n).view(np.int64) + rng.integers(-6, 7, n)
        v = np.abs(v.view(np.float64))
        v[::97] = np.ldexp(rng.uniform(0.5, 1.0, len(v[::97])), -1060)   # subnormal
    return v.reshape(shape)


def _wrong(got, a):
    exact = np.log(a.astype(np.longdouble)).astype(np.float32)
    return int(np.sum((got != exact) & (got != np.log(a).astype(np.float32))))


@pytest.mark.parametrize("kind", ["exponents", "near_one", "ordinary", "edges"])
def test_logarithms_bit_for_bit(q, kind):
    import torch
    rng = np.random.default_rng(len(kind))
    A, B = _values(rng, kind, (N_T, N_S)), _values(rng, kind, (N_T - 1, N_S))
    ptr = np.arange(N_S + 1, dtype=np.int32)
    ctx = q.qsel_create_bt(N_S, N_T, ptr, ptr[:-1].copy(), A, -B, n_parts=2, overlap=1, n_samples=2,
                           precision=q.QSEL_MIXED)
    F = torch.empty((N_S * N_T, q.QSEL_CV_FEATURES), dtype=torch.float32, device="cuda")
    q.qsel_cv_features(ctx, 1, F)
    F = F.cpu().numpy().reshape(N_T, N_S, -1)
    assert _wrong(F[:, :, 0], A) == 0
    two = np.zeros((2, N_T, N_S))
    two[0, 1:], two[1, :-1] = B, B
    top = np.maximum(np.sort(two, 0)[::-1], 1e-30)
    assert _wrong(F[:, :, 1], top[0]) == 0
    assert _wrong(F[:, :, 2], top[1]) == 0
    assert _wrong(F[:, :, 3:9], np.full((N_T, N_S, 6), 1e-30)) == 0
