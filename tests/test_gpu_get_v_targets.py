"""chicle_get_v into every kind of array that the copy behind it takes: the caller's own device memory, the same at an odd
address, pinned host memory passed as device memory (both are addressable), host memory; a foreign length is refused. The same
bits everywhere."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1909_04885_b200 import binding  # noqa: E402
from test_gpu_parity import tiny_csr  # noqa: E402


def test_targets():
    import torch
    w = tiny_csr(300, 77, seed=3, K=3)
    glm = binding.from_workload(w)
    try:
        glm.partition(3, 1)
        glm.cocoa_round(0, 3.0)
        want = glm.get_v().copy()
        assert np.abs(want).max() > 0
        d = glm.dim
        raw = torch.zeros(4 * d + 8, dtype=torch.uint8, device="cuda")
        pinned = torch.zeros(d, dtype=torch.float32).pin_memory()
        torch.cuda.synchronize()
        for off in (0, 1, 2, 4):
            raw.zero_()
            torch.cuda.synchronize()
            glm._check(glm._lib.chicle_get_v(glm._h, C.c_void_p(raw.data_ptr() + off), d, binding.MEM_DEVICE))
            assert np.array_equal(raw.cpu().numpy()[off:off + 4 * d].copy().view(np.float32), want)
            assert raw[off + 4 * d:].sum().item() == 0 and raw[:off].sum().item() == 0
        glm.get_v(pinned)
        torch.cuda.synchronize()
        assert np.array_equal(pinned.numpy(), want)
        assert glm._lib.chicle_get_v(glm._h, C.c_void_p(raw.data_ptr()), d - 1, binding.MEM_DEVICE) == binding.ERR_INVALID_ARG
    finally:
        glm.close()
