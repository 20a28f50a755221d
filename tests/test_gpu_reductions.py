"""The reductions at the edges of their groups: pattern sums of fewer rows than
one slice up to more than one run per block, more slabs than the trace
combination has threads, and PCG dots of fewer partial rows than row groups and
of more than one batch of them.  The exact one-part result and the injected
RBMC result of the binary64 form against the oracle, 1e-10 relative as for the
other parity tests; the PCG's samples to their residual."""
import numpy as np
import pytest

import qsel_inputs as qi
from oracle import qsel_oracle as o
from tests.models import theta as mk_theta
from tests.test_gpu_parity import q, rel_err  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _make(q, m, n_t, parts=1, k=4, **kw):
    mesh = qi.grid_mesh(m)
    mask = qi.obs_mask(m * m * n_t, 0.3, 4)
    th = mk_theta(0.5, 1.2, 0.8)
    model = o.model_from_csr(m * m, n_t, mesh.c_diag, mesh.g_rowptr, mesh.g_col, mesh.g_val, mask, 0.5)
    ctx = q.qsel_create(m * m, n_t, mesh.c_diag, mesh.g_rowptr, mesh.g_col, mesh.g_val, mask, 0.5, th,
                        n_parts=parts, overlap=min(1, parts - 1), n_samples=k, seed=3, precision=q.QSEL_FP64, **kw)
    return ctx, model, th


@pytest.mark.parametrize("m,n_t", [(3, 2), (3, 300), (6, 4), (17, 3), (23, 2)])
def test_pattern_sums_and_traces(q, m, n_t):
    ctx, model, th = _make(q, m, n_t)
    v_ex, t_ex = o.exact_selinv(o.precision(model, th), o.precision_derivatives(model, th))
    assert rel_err(ctx.diag_inv(), v_ex) <= 1e-10
    assert rel_err(ctx.trace_grads(), t_ex) <= 1e-10


@pytest.mark.parametrize("m,n_t,k", [(3, 4, 5), (16, 6, 64), (24, 12, 70)])
def test_pcg_dots(q, m, n_t, k):
    ctx, model, th = _make(q, m, n_t, parts=2, k=k, pcg_tol=1e-10)
    ctx.diag_inv()
    X = q.qsel_debug_get_samples(ctx)
    Q = o.precision(model, th)
    R = o.rhs(model, th, 3, k)
    res = np.linalg.norm(R - Q @ X, axis=0) / np.linalg.norm(R, axis=0)
    assert res.max() <= 1e-9
    assert ctx.stats()["pcg_max_rel_residual"] <= 1e-10
