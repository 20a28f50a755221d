"""The pivot chain of the mixed form's blocked sweep (csrc/sweep_chain.cu) for
every panel shape: one to four pivots in the only panel, full panels with a
ragged last one, for both pivot precisions and with several matrices a launch,
against the CPU oracle's exact selected inverse.

Tolerance: the mixed form's stated 5e-4 relative per result (n_s <= 1600)."""
import numpy as np
import pytest

import qsel_inputs as qi
from oracle import qsel_oracle as o
from tests.models import grid_model, theta as mk_theta
from tests.test_gpu_parity import q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b)) / np.abs(np.asarray(b))))


@pytest.mark.parametrize("fp64_pivots", [False, True])
@pytest.mark.parametrize("m", [7, 11, 13, 16, 17, 19, 21, 23])   # 1, 2, 3, 4, 5, 6, 7, 9 tiles
def test_panels(q, m, fp64_pivots):
    n_t = 3
    model, mesh, th = grid_model(m, n_t, 0.3), qi.grid_mesh(m), mk_theta(0.5, 1.2, 0.85)
    ctx = q.qsel_create(model.n_s, n_t, mesh.c_diag, mesh.g_rowptr, mesh.g_col, mesh.g_val, model.obs_mask,
                        model.sigma, th, n_parts=1, overlap=0, n_samples=2, precision=q.QSEL_MIXED,
                        pivot_precision=q.QSEL_PIVOT_FP64 if fp64_pivots else q.QSEL_PIVOT_DOUBLE_FLOAT)
    v_or, t_or = o.exact_selinv(o.precision(model, th), o.precision_derivatives(model, th))
    assert _rel(ctx.diag_inv(), v_or) <= 5e-4
    assert _rel(ctx.trace_grads(), t_or) <= 5e-4


@pytest.mark.parametrize("parts", [2, 5])
def test_several_matrices(q, parts):
    m, n_t, k = 18, 3 * parts, 8
    model, mesh, th = grid_model(m, n_t, 0.3), qi.grid_mesh(m), mk_theta(0.5, 1.2, 0.85)
    ctx = q.qsel_create(model.n_s, n_t, mesh.c_diag, mesh.g_rowptr, mesh.g_col, mesh.g_val, model.obs_mask,
                        model.sigma, th, n_parts=parts, overlap=1, n_samples=k, precision=q.QSEL_MIXED)
    X = qi.seeded_normal((model.n, k), 3)
    q.qsel_debug_set_samples(ctx, X)
    v_or, t_or, _ = o.rbmc(model, th, o.balanced_slab_start(n_t, parts), 1, X)
    assert _rel(ctx.diag_inv(), v_or) <= 5e-4
    assert _rel(ctx.trace_grads(), t_or) <= 5e-4
