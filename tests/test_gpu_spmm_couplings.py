"""The SpMM over blocks whose couplings live on a smaller pattern than the
diagonal blocks: rows of more than 32 entries (two batches of a warp), couplings
on none, one and several of them, in the first and in the second batch.  Through
the Lanczos sampler (its only operator is this product) against the oracle's,
1e-10 of the largest entry as for its other tests."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import qsel_lanczos as lz
from tests.test_gpu_models import bt_inputs, q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_s,k", [(40, 8), (40, 70), (64, 130)])
def test_sparse_couplings(q, n_s, k):
    n_t, rng = 4, np.random.default_rng(n_s)
    Q = np.zeros((n_s * n_t, n_s * n_t))
    for t in range(n_t):
        a = slice(t * n_s, (t + 1) * n_s)
        M = rng.normal(0, 1, (n_s, n_s)) / np.sqrt(n_s)
        Q[a, a] = 3.0 * np.eye(n_s) + M @ M.T
        if t + 1 < n_t:
            B = np.zeros((n_s, n_s))
            B[1, 1], B[n_s - 1, n_s - 1] = 0.3, -0.2   # row 0 has no coupling
            for i, j in ((2, 3), (2, n_s - 2), (5, n_s - 1), (n_s - 3, n_s - 2)):
                B[i, j] = B[j, i] = rng.uniform(-0.4, 0.4)
            b = slice((t + 1) * n_s, (t + 2) * n_s)
            Q[a, b] = Q[b, a] = B
    assert np.linalg.eigvalsh(Q)[0] > 0.5
    Q = sp.csr_matrix(Q)
    rowptr, col, diag, off, dd, do = bt_inputs(Q, [], n_s, n_t)
    ctx = q.qsel_create_bt(n_s, n_t, rowptr, col, diag, off, dd, do, n_parts=2, overlap=1, n_samples=k, seed=5,
                           precision=q.QSEL_FP64, lanczos_steps=10, precond_block=16)
    ctx.diag_inv()
    X = q.qsel_debug_get_samples(ctx)
    X_or, _, _ = lz.sample_q(Q, 5, k, 10, 16)
    assert np.max(np.abs(X - X_or)) <= 1e-10 * np.max(np.abs(X_or))
