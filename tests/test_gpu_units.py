"""The binary64 form on unknowns in different units: Q and D Q D with D
diagonal over 10^-6 .. 10^6 (entries of Q over 10^24).

D of powers of two scales every operand and every result exactly, so the
selected inverse, the correction, the samples, the block applies and the
gradient's K^-1 must give the same bits but for the exponents (diag / d^2, x / d,
equal traces).  D of other values is compared with the oracle on the unscaled
matrix at the form's 1e-10 relative."""
import numpy as np
import pytest
import scipy.sparse as sp

import qsel_inputs as qi
from oracle import qsel_oracle as o
from tests.models import grid_model, theta as mk_theta
from tests.test_gpu_parity import q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


class Blocks:
    """A separable model's Q and dQ as user-given blocks, scaled by d (n_s) and g (n_t)."""

    def __init__(self, m, n_t, seed=3):
        self.n_s, self.n_t = m * m, n_t
        self.model, th = grid_model(m, n_t, 0.3), mk_theta(0.7, 1.2, 0.85)
        self.Q, self.dQ = o.precision(self.model, th), o.precision_derivatives(self.model, th)
        n_s = self.n_s
        pat = sum(abs(M[:n_s, :n_s]) for M in [self.Q] + list(self.dQ))
        if n_t > 1:
            pat = pat + sum(abs(M[:n_s, n_s:2 * n_s]) for M in [self.Q] + list(self.dQ))
        pat = sp.csr_matrix(pat + sp.identity(n_s))
        pat.sort_indices()
        self.rowptr, self.col = pat.indptr.astype(np.int32), pat.indices.astype(np.int32)
        self.row = np.repeat(np.arange(n_s), np.diff(self.rowptr))

    def values(self, M, d, g):
        n_s, n_t = self.n_s, self.n_t
        M = sp.csr_matrix(M)
        w = d[self.row] * d[self.col]

        def block(t, u):
            B = M[t * n_s:(t + 1) * n_s, u * n_s:(u + 1) * n_s].toarray()
            B = 0.5 * (B + B.T)
            return B[self.row, self.col] * w * (g[t] * g[u])
        return (np.array([block(t, t) for t in range(n_t)]),
                np.array([block(t, t + 1) for t in range(n_t - 1)]).reshape(n_t - 1, len(self.col)))

    def context(self, q, d, g, **kw):
        A, B = self.values(self.Q, d, g)
        parts = [self.values(M, d, g) for M in self.dQ]
        return q.qsel_create_bt(self.n_s, self.n_t, self.rowptr, self.col, A, B, np.array([p[0] for p in parts]),
                                np.array([p[1] for p in parts]), precision=q.QSEL_FP64, **kw)


def _units(n_s, n_t, seed, powers=True):
    rng = np.random.default_rng(seed)
    if powers:
        return 2.0 ** rng.integers(-20, 21, n_s), 2.0 ** rng.integers(-3, 4, n_t)
    return 10.0 ** rng.uniform(-6.0, 6.0, n_s), 10.0 ** rng.uniform(-1.0, 1.0, n_t)


def _rel(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b)) / np.abs(np.asarray(b))))


@pytest.mark.parametrize("m,n_t,chain", [(7, 1, "forward"), (13, 4, "forward"), (13, 5, "two_ended"), (23, 3, "two_ended")])
def test_exact_selected_inverse(q, m, n_t, chain):
    b = Blocks(m, n_t)
    kw = dict(n_parts=1, overlap=0, n_samples=2,
              chain=q.QSEL_CHAIN_FORWARD if chain == "forward" else q.QSEL_CHAIN_TWO_ENDED)
    one = b.context(q, np.ones(b.n_s), np.ones(n_t), **kw)
    v1, t1 = one.diag_inv(), q.qsel_trace_grads_n(one, 3)
    v_or, t_or = o.exact_selinv(b.Q, b.dQ)
    assert _rel(v1, v_or) <= 1e-10
    for powers in (False, True):
        d, g = _units(b.n_s, n_t, 11, powers)
        u = np.kron(g, d)
        ctx = b.context(q, d, g, **kw)
        v, t = ctx.diag_inv() * u * u, q.qsel_trace_grads_n(ctx, 3)
        assert _rel(v, v_or) <= 1e-10
        assert _rel(t, t_or) <= 1e-10
    assert np.array_equal(v, v1) and np.array_equal(t, t1)


@pytest.mark.parametrize("m,n_t,parts,overlap,k", [(8, 7, 2, 2, 3), (13, 8, 3, 1, 70)])
def test_correction_with_injected_samples(q, m, n_t, parts, overlap, k):
    b = Blocks(m, n_t)
    kw = dict(n_parts=parts, overlap=overlap, n_samples=k)
    X = qi.seeded_normal((b.n_s * n_t, k), 5)

    def run(d, g):
        u = np.kron(g, d)
        ctx = b.context(q, d, g, **kw)
        q.qsel_debug_set_samples(ctx, X / u[:, None])
        return ctx.diag_inv() * u * u, q.qsel_trace_grads_n(ctx, 3)

    v1, t1 = run(np.ones(b.n_s), np.ones(n_t))
    for powers in (False, True):
        v, t = run(*_units(b.n_s, n_t, 12, powers))
        assert _rel(v, v1) <= 1e-10
        assert _rel(t, t1) <= 1e-10
    assert np.array_equal(v, v1) and np.array_equal(t, t1)


@pytest.mark.parametrize("m,n_t,k,block", [(9, 4, 70, 16), (13, 3, 33, 32), (13, 3, 130, 64)])
def test_block_applies_and_lanczos_samples(q, m, n_t, k, block):
    b = Blocks(m, n_t)
    kw = dict(n_parts=1, overlap=0, n_samples=k, precond_block=block)
    R = qi.seeded_normal((b.n_s * n_t, k), 9)

    def apply(d, g):
        u = np.kron(g, d)[:, None]
        return q.qsel_debug_apply_precond(b.context(q, d, g, **kw), R * u) * u

    def samples(d, g):
        ctx = b.context(q, d, g, n_parts=n_t, overlap=0, n_samples=k, precond_block=block, lanczos_steps=12, seed=4)
        ctx.diag_inv()
        return q.qsel_debug_get_samples(ctx) * np.kron(g, d)[:, None]

    for f in (apply, samples):
        z1 = f(np.ones(b.n_s), np.ones(n_t))
        for powers in (False, True):
            z = f(*_units(b.n_s, n_t, 13, powers))
            # per column, against the column's largest entry of the unscaled unknowns
            assert np.max(np.abs(z - z1) / np.abs(z1).max(0)) <= 1e-10
        assert np.array_equal(z, z1)


def test_gradient_term_from_the_dense_inverse(q):
    """K = kappa^2 C + G with C = D^2 C0 and G = D G0 D: tr(K^-1 C) is K0's."""
    m, n_t = 15, 3
    mesh, th = qi.grid_mesh(m), mk_theta(0.5, 1.3, 0.9)
    n_s = m * m
    mask = qi.obs_mask(n_s * n_t, 0.3, 1)
    row = np.repeat(np.arange(n_s), np.diff(mesh.g_rowptr))

    def prior(d):
        ctx = q.qsel_create(n_s, n_t, mesh.c_diag * d * d, mesh.g_rowptr, mesh.g_col,
                            mesh.g_val * d[row] * d[mesh.g_col], mask, 0.5, th, precision=q.QSEL_FP64, n_parts=1,
                            overlap=0, n_samples=2, pcg_tol=0.5)
        q.qsel_set_data(ctx, qi.seeded_normal((int(mask.sum()), 1), 7)[:, 0])
        return np.asarray(q.qsel_loglik_grad(ctx, with_terms=True)[1][0])

    p1 = prior(np.ones(n_s))
    assert _rel(prior(_units(n_s, 1, 14, False)[0]), p1) <= 1e-10
    assert np.array_equal(prior(_units(n_s, 1, 14)[0]), p1)


def test_zero_rows_and_far_exponents(q):
    """Rows of zeros beside rows of 2^+-300, diagonal blocks: the inverse's
    diagonal is exact, whatever the shifts of the other entries."""
    n_s, n_t = 130, 3
    rng = np.random.default_rng(5)
    e = rng.integers(-300, 301, (n_t, n_s))
    A = 2.0 ** (2 * e)
    ptr = np.arange(n_s + 1, dtype=np.int32)
    ctx = q.qsel_create_bt(n_s, n_t, ptr, ptr[:-1].copy(), A, np.zeros((n_t - 1, n_s)), precision=q.QSEL_FP64,
                           n_parts=1, overlap=0, n_samples=2)
    assert np.array_equal(ctx.diag_inv(), (1.0 / A).reshape(-1))
