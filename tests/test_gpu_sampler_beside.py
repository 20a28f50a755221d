"""The sampler beside the first wave's dense part (its own stream) against the
sequential order that a profiled pass keeps: the same launches on the same
data, so the same bits, on the first pass and on repeated ones."""
import numpy as np
import pytest

from tests.test_gpu_models import Diff
from tests.test_gpu_parity import Case, q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["pcg_fp64", "lanczos_fp64", "lanczos_mixed"])
def test_beside_equals_sequential(q, kind):
    def case(profile):
        if kind == "pcg_fp64":
            return Case(q, "ragged13", precision=q.QSEL_FP64, profile_kernels=profile)
        prec = q.QSEL_FP64 if kind == "lanczos_fp64" else q.QSEL_MIXED
        return Diff(q, "diff9_ragged", precision=prec, profile_kernels=profile)

    ref = case(1)
    v_ref, t_ref = ref.ctx.diag_inv(), ref.ctx.trace_grads()
    c = case(0)
    for _ in range(3):
        assert np.array_equal(c.ctx.diag_inv(), v_ref)
        assert np.array_equal(c.ctx.trace_grads(), t_ref)
        q.qsel_set_theta(c.ctx, c.theta)
