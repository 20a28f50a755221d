"""A binary64 Lanczos context on a device that is nearly full: memory for the
plain dense working sets and the sampler's buffers, but not for the digit
products' scratch on top.  The context has to leave the scratch out (the
CUDA-core products serve) instead of failing in the sampler's allocation."""
import ctypes

import numpy as np
import pytest

from tests.test_gpu_models import DIFF, Diff, q  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

# 1024-node blocks, two parts of three slabs; 420 steps: about 100 MB of sampler buffers
DIFF["tight32"] = (32, 4, 0.5, 1.5, 0.8, 0.3, 0.5, 2, 1, 64)


def _digit_scratch(n_pad, ld, T):
    rows = max(n_pad, ld)
    return 2 * (16 * rows * n_pad + 4 * rows) + 4 * (T + 2) * n_pad + 2 * 16 * n_pad * 64 + 8 * n_pad


def test_lanczos_with_little_memory(q):
    import torch

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def run():
        f0 = free()
        c = Diff(q, "tight32", precision=q.QSEL_FP64, lanczos_steps=420)
        v, t = c.ctx.diag_inv(), c.ctx.trace_grads()
        used = f0 - free()
        c.ctx.close()
        return v, t, used

    run()   # the kernels' code is on the device from here on
    v1, t1, used = run()
    torch.cuda.empty_cache()
    target = used - _digit_scratch(1024, 64, 3)   # two slots: half of their scratch is missing
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    hold = ctypes.c_void_p()
    assert rt.cudaMalloc(ctypes.byref(hold), ctypes.c_size_t((free() - target) >> 21 << 21)) == 0
    try:
        assert abs(free() - target) <= 8 << 20
        v, t, _ = run()
    finally:
        assert rt.cudaFree(hold) == 0
    # the same samples; dense products on other kernels
    assert np.max(np.abs(v - v1) / v1) <= 1e-10
    assert np.max(np.abs(np.asarray(t) - t1) / np.abs(t1)) <= 1e-10
