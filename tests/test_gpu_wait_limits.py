"""The bounded waits of the binary64 form's tensor-core kernels, run out
without a GPU fault: the test hook makes the products' producer issue no load
(their waits end after 2e6 cycles, about 1 ms).  The call reports QSEL_ETIMEOUT, and the next one on the same context, with
the limits restored, is right: no error word is left over."""
import numpy as np
import pytest

import qsel_inputs as qi
from oracle import qsel_hyper as oh
from oracle import qsel_oracle as o
from tests.test_gpu_parity import Case, q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

ETIMEOUT = 6


def _case(q, **kw):
    return Case(q, "grid16_nt8", precision=q.QSEL_FP64, **kw)


def _rel(a, b):
    return float(np.max(np.abs(np.asarray(a) - np.asarray(b)) / np.abs(np.asarray(b))))


def _times_out(q, call, skip_loads, cycles):
    q.qsel_debug_tc_wait(skip_loads, cycles)
    try:
        with pytest.raises(q.QselError) as ei:
            call()
    finally:
        q.qsel_debug_tc_wait(False, 0)
    assert ei.value.status == ETIMEOUT


def test_products_then_posterior_mean(q):
    c = _case(q, parts=1, overlap=0)
    y = qi.seeded_normal((int(c.mask.sum()), 1), 7)[:, 0]
    q.qsel_set_data(c.ctx, y)
    _times_out(q, c.ctx.diag_inv, True, 2_000_000)
    # the mean's solve has not timed out
    mu, mu_or = q.qsel_posterior_mean(c.ctx), oh.posterior_mean(c.model, c.theta, y)
    assert np.max(np.abs(mu - mu_or)) <= 1e-7 * np.max(np.abs(mu_or))
    _times_out(q, c.ctx.diag_inv, True, 2_000_000)
    v_ex, _ = o.exact_selinv(o.precision(c.model, c.theta), o.precision_derivatives(c.model, c.theta))
    assert _rel(c.ctx.diag_inv(), v_ex) <= 1e-10


def test_products_beside_a_sampler(q):
    c = _case(q)
    _times_out(q, c.ctx.diag_inv, True, 2_000_000)
    X = qi.seeded_normal((c.n_s * c.n_t, c.k), 99)
    q.qsel_debug_set_samples(c.ctx, X)
    v_or, _, _ = o.rbmc(c.model, c.theta, c.slab_start, c.n_l, X)
    assert _rel(c.ctx.diag_inv(), v_or) <= 1e-10
