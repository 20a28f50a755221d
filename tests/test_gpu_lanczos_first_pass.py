"""The Lanczos sampler's first pass on device memory that held something else
before: its buffers are allocated in the call, and what it takes as zero has
to be cleared on the sampler's own stream.  The memory is filled with NaN
patterns and freed, so that the context's allocations receive it."""
import ctypes

import numpy as np
import pytest

from tests.test_gpu_models import Diff, q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _leave_nan_patterns():
    """Freed device memory full of NaNs: blocks of many small sizes from the
    driver's own pools, every other one kept until the end so that the pools
    stay, and the kept ones (to be freed by the caller)."""
    import torch
    torch.cuda.synchronize()
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    kept, freed = [], []
    for size in (512, 1024, 2048, 4096, 16384, 65536, 1 << 20):
        for i in range(400 if size < 65536 else 40):
            p = ctypes.c_void_p()
            assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0
            assert rt.cudaMemset(p, 0xFF, ctypes.c_size_t(size)) == 0
            (kept if i % 2 else freed).append(p)
    assert rt.cudaDeviceSynchronize() == 0
    for p in freed:
        assert rt.cudaFree(p) == 0
    return rt, kept


@pytest.mark.parametrize("name", ["diff9_ragged", "diff24_panels"])
def test_first_pass_on_used_memory(q, name):
    ref = Diff(q, name, precision=q.QSEL_FP64)
    v_ref, t_ref = ref.ctx.diag_inv(), ref.ctx.trace_grads()
    assert np.isfinite(v_ref).all()
    ref.ctx.close()
    rt, kept = _leave_nan_patterns()
    try:
        c = Diff(q, name, precision=q.QSEL_FP64)
        # the same launches on the same data: the same bits
        assert np.array_equal(c.ctx.diag_inv(), v_ref)
        assert np.array_equal(c.ctx.trace_grads(), t_ref)
    finally:
        for p in kept:
            rt.cudaFree(p)
