"""The tensor-core Kronecker apply over the tile shapes that short axes take:
grids and slab counts that fill a tile from one, two or three axes, with and
without padding, against the oracle's operator in binary64 on the same (rounded)
input.  Tolerance as for the other mixed applies: 2e-5 of the largest entry,
binary32 accuracy of six contractions."""
import numpy as np
import pytest

import qsel_inputs as qi
from oracle import qsel_kron as kr
from tests.test_gpu_kron import _grid_ctx
from tests.test_gpu_parity import q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n_t,k", [(4, 4, 64), (36, 4, 64), (20, 12, 64), (12, 24, 192), (16, 16, 256),
                                     (8, 36, 320), (4, 132, 64)])
def test_short_axes(q, m, n_t, k):
    ctx, model, th = _grid_ctx(q, m, n_t, k, preconditioner=q.QSEL_PRECOND_KRON, precision=q.QSEL_MIXED)
    R = qi.seeded_normal((model.n, k), 23).astype(np.float32).astype(np.float64)
    Z = q.qsel_debug_apply_precond(ctx, R)
    Z_or = kr.preconditioner_inverse(model, th) @ R
    err = np.max(np.abs(Z - Z_or)) / np.max(np.abs(Z_or))
    print(f"m={m} n_t={n_t} k={k}: {err:.2e}")
    assert err <= 2e-5
