"""Binary64 dense products as exact bf16 digit products (csrc/oz.cuh): the
selected inverse, the correction and the hyperparameter gradient in QSEL_FP64
at the sizes where the tiles can go wrong -- one ragged 64 tile, an odd number
of them (half of a 128-row tile empty), K past one and several exact sums of
128, more sample columns than nodes -- against the CPU oracle.

Tolerance: the binary64 form's stated 1e-10 relative per result."""
import numpy as np
import pytest

import qsel_inputs as qi
from oracle import qsel_hyper as oh
from oracle import qsel_oracle as o
from tests.models import grid_model, theta as mk_theta
from tests.test_gpu_parity import q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _ctx(q, model, mesh, th, **kw):
    return q.qsel_create(model.n_s, model.n_t, mesh.c_diag, mesh.g_rowptr, mesh.g_col, mesh.g_val, model.obs_mask,
                         model.sigma, th, precision=q.QSEL_FP64, **kw)


def _rel(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b)) / np.abs(np.asarray(b))))


@pytest.mark.parametrize("m,n_t", [(2, 3), (8, 2), (9, 4), (11, 5), (13, 3), (17, 4), (23, 3)])
def test_exact_selected_inverse(q, m, n_t):
    model, mesh, th = grid_model(m, n_t, 0.2), qi.grid_mesh(m), mk_theta(0.3, 1.3, 0.9)
    ctx = _ctx(q, model, mesh, th, n_parts=1, overlap=0, n_samples=2)
    Q, dQ = o.precision(model, th), o.precision_derivatives(model, th)
    v_or, t_or = o.exact_selinv(Q, dQ)
    assert _rel(ctx.diag_inv(), v_or) <= 1e-10
    assert _rel(ctx.trace_grads(), t_or) <= 1e-10


@pytest.mark.parametrize("m,n_t,parts,overlap,k", [(4, 9, 3, 1, 130), (8, 7, 2, 2, 3), (12, 8, 3, 1, 70)])
def test_correction_with_injected_samples(q, m, n_t, parts, overlap, k):
    model, mesh, th = grid_model(m, n_t, 0.2), qi.grid_mesh(m), mk_theta(0.4, 0.8, 0.85)
    ctx = _ctx(q, model, mesh, th, n_parts=parts, overlap=overlap, n_samples=k)
    X = qi.seeded_normal((model.n, k), 5)
    q.qsel_debug_set_samples(ctx, X)
    v_or, t_or, _ = o.rbmc(model, th, o.balanced_slab_start(n_t, parts), overlap, X)
    assert _rel(ctx.diag_inv(), v_or) <= 1e-10
    assert _rel(ctx.trace_grads(), t_or) <= 1e-10


@pytest.mark.parametrize("scale", [1e-120, 1e120])
def test_scaled_blocks(q, scale):
    """tau scales Q_x and 1/sigma^2 the observations alike, so diag(Q^-1) scales
    by 1 / scale: row exponents far from zero, with results in range."""
    m, n_t = 9, 3
    model, mesh, th = grid_model(m, n_t, 0.2), qi.grid_mesh(m), mk_theta(0.3, 1.0, 0.9)
    v_or, _ = o.exact_selinv(o.precision(model, th), o.precision_derivatives(model, th))
    model.sigma /= np.sqrt(scale)
    ctx = _ctx(q, model, mesh, (th[0], th[1] + np.log(scale), th[2]), n_parts=1, overlap=0, n_samples=2)
    # log(scale) carries 4e-14 relative of its own into tau
    assert _rel(ctx.diag_inv() * scale, v_or) <= 1e-10


def test_gradient_term_from_the_dense_inverse(q):
    """K^-1 of the hyperparameter gradient runs the same sweep on one matrix."""
    m, n_t = 15, 3
    model, mesh, th = grid_model(m, n_t, 0.3), qi.grid_mesh(m), mk_theta(0.3, 1.3, 0.9)
    ctx = _ctx(q, model, mesh, th, n_parts=1, overlap=0, n_samples=2)
    q.qsel_set_data(ctx, qi.seeded_normal((int(model.obs_mask.sum()), 1), 7)[:, 0])
    _, (prior, _, _) = q.qsel_loglik_grad(ctx, with_terms=True)
    assert _rel(prior, oh.prior_logdet_grad(model, th)) <= 1e-10


@pytest.mark.parametrize("m,n_t,k,block", [(5, 3, 10, 64), (9, 4, 70, 32), (8, 5, 130, 16), (13, 3, 200, 64)])
def test_block_jacobi_apply(q, m, n_t, k, block):
    """Z = P^-1 R block by block: one ragged 64-row tile, rows past n, blocks
    smaller than the tile, one and several 128-column chunks."""
    model, mesh, th = grid_model(m, n_t, 0.3), qi.grid_mesh(m), mk_theta(0.4, 1.1, 0.8)
    ctx = _ctx(q, model, mesh, th, n_parts=1, overlap=0, n_samples=k, precond_block=block)
    R = qi.seeded_normal((model.n, k), 9) * np.logspace(-6, 6, k)
    Z = q.qsel_debug_apply_precond(ctx, R)
    Q = o.precision(model, th).toarray()
    ref = np.concatenate([np.linalg.solve(Q[a:a + block, a:a + block], R[a:a + block]) for a in range(0, model.n, block)])
    # per column, against the column's largest entry: the digits are scaled by it
    assert np.max(np.abs(Z - ref) / np.abs(ref).max(0)) <= 1e-11
