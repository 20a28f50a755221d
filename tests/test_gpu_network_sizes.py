"""The control variate's kernels at the edges of their launches: one and two
samples per thread in the forward pass, the tile groups of the gradient's
reduction, buffers that start on four bytes, and the features of models whose
blocks repeat, or differ, from slab to slab.

Tolerances: as for the other control-variate tests, 1e-6 relative (1e-5
absolute) for the features, which are binary64 values rounded to float, and
1e-4 of the largest value for FP32 sums of at most 64 terms; the gradient sums
its tiles in binary64."""
import math

import numpy as np
import pytest

import qsel_inputs as qi
from oracle import qsel_mlp as om
from oracle import qsel_oracle as o
from tests.test_gpu_cv import ORDER, _as_used, _dev, _flat, _params
from tests.test_gpu_models import bt_inputs, random_bt
from tests.test_gpu_parity import mk_theta, q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _unaligned(n):
    """A float buffer of n values that starts 4 bytes past a 16-byte boundary."""
    import torch
    return torch.empty(n + 1, dtype=torch.float32, device="cuda")[1:]


@pytest.mark.parametrize("n", [1, 255, 257, 256 * 152, 256 * 152 + 1, 512 * 152 + 513])
@pytest.mark.parametrize("aligned", [True, False])
def test_forward_sizes(q, n, aligned):
    import torch
    P = _as_used(_params(1))
    cv = q.qsel_cv_create(0)
    q.qsel_cv_set_params(cv, _flat(P))
    X = np.random.default_rng(n).normal(0, 1.5, (n, 14)).astype(np.float32)
    Xd = _dev(X)
    if not aligned:
        Xu = _unaligned(n * 14)
        Xu.copy_(Xd.reshape(-1))
        Xd = Xu
    y = torch.full((n + 1,), 7.0, dtype=torch.float32, device="cuda")
    q.qsel_cv_predict(cv, Xd, y, n)
    y_or, _ = om.forward(P, X.astype(np.float64), bf16=True)
    assert np.max(np.abs(y[:n].cpu().numpy() - y_or)) <= 1e-4 * max(1.0, np.max(np.abs(y_or)))
    assert float(y[n]) == 7.0


@pytest.mark.parametrize("n", [65, 64 * 63 + 1, 64 * 70, 256 * 152 + 300])
def test_gradient_sizes(q, n):
    P = _as_used(_params(3))
    cv = q.qsel_cv_create(0)
    q.qsel_cv_set_params(cv, _flat(P))
    rng = np.random.default_rng(4)
    X = rng.normal(0, 1.5, (n, 14)).astype(np.float32).astype(np.float64)
    t = rng.normal(0, 1, n).astype(np.float32).astype(np.float64)
    g, loss = q.qsel_cv_grad(cv, _dev(X), _dev(t), n)
    loss_or, g_or = om.loss_and_grad(P, X, t, bf16=True)
    assert abs(loss - loss_or) <= 1e-5 * loss_or
    off = 0
    for k in ORDER:
        ref = np.ravel(g_or[k])
        got = g[off:off + ref.size]
        off += ref.size
        assert np.max(np.abs(got - ref)) <= 1e-4 * np.max(np.abs(ref)), k


@pytest.mark.parametrize("n_t,aligned", [(1, True), (2, True), (16, True), (17, False), (35, True)])
def test_features_over_slab_ranges(q, n_t, aligned):
    m, sigma, theta = 7, 0.5, mk_theta(0.6, 1.3, 0.8)
    mesh = qi.grid_mesh(m)
    n = m * m * n_t
    mask = qi.obs_mask(n, 0.3, 1)
    model = o.model_from_csr(m * m, n_t, mesh.c_diag, mesh.g_rowptr, mesh.g_col, mesh.g_val, mask, sigma)
    parts = 1 if n_t < 4 else 3
    ss = qi.balanced_slab_start(n_t, parts)
    ctx = q.qsel_create(m * m, n_t, mesh.c_diag, mesh.g_rowptr, mesh.g_col, mesh.g_val, mask, sigma, theta,
                        n_parts=parts, slab_start=ss, overlap=min(1, parts - 1), n_samples=4, seed=1)
    F = _unaligned(n * 14) if not aligned else _dev(np.zeros(n * 14))
    q.qsel_cv_features(ctx, 1, F)
    np.testing.assert_allclose(F.cpu().numpy().reshape(n, 14), om.features(model, theta, ss, 1), rtol=1e-6, atol=1e-5)


def test_features_of_blocks_that_differ(q):
    """User-given blocks, different in every slab: no slab may take another's."""
    n_s, n_t, Q, dQs = random_bt(n_t=19)
    rowptr, col, diag, off, dd, do = bt_inputs(Q, dQs, n_s, n_t)
    ctx = q.qsel_create_bt(n_s, n_t, rowptr, col, diag, off, dd, do, n_parts=1, n_samples=4)
    F = _dev(np.zeros(n_s * n_t * 14))
    q.qsel_cv_features(ctx, 1, F)
    Q = Q.tocsr()
    ref = np.zeros((n_s * n_t, 9))
    for r in range(n_s * n_t):
        c, v = Q.indices[Q.indptr[r]:Q.indptr[r + 1]], Q.data[Q.indptr[r]:Q.indptr[r + 1]]
        top = np.sort(np.abs(v[(c != r) & (v != 0.0)]))[::-1][:8]
        ref[r, 0] = math.log(v[c == r][0])
        ref[r, 1:] = np.log(np.maximum(np.pad(top, (0, 8 - len(top))), 1e-30))
    np.testing.assert_allclose(F.cpu().numpy().reshape(-1, 14)[:, :9], ref, rtol=1e-6, atol=1e-5)
