"""Host arrays that a call reads while it runs (the header's words): a caller that passes pinned memory, which a copy reads only
when the stream gets there, may overwrite it as soon as the call has returned."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from parity_util import make_pair, rel_l2  # noqa: E402
from test_gpu_record_slots import sparse  # noqa: E402


@pytest.mark.parametrize("K", [40, 4000])
def test_pinned_budgets_and_flags(K):
    import torch
    w = sparse("hinge", 12000, 500, 5, K, 0.5, seed=K)
    orc, glm = make_pair(w)
    try:
        orc.partition(K, 1)
        glm.partition(K, 1)
        steps = np.array([k % 4 for k in range(K)], np.int64)
        pinned = torch.from_numpy(steps.copy()).pin_memory()
        keep = torch.from_numpy((np.arange(K) % 2).astype(np.uint8)).pin_memory()
        out = torch.zeros(glm.n_coord, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        torch.cuda._sleep(40_000_000)  # the stream is busy when the calls return
        glm.cocoa_round(0, float(K), steps=pinned.numpy())
        pinned.fill_(3)
        torch.cuda._sleep(40_000_000)
        glm.export_state_of(keep.numpy(), out)
        keep.fill_(1)
        orc.cocoa_round(0, float(K), steps=steps)
        a = glm.get_alpha()
        assert rel_l2(a, orc.state) <= 1e-4
        assert np.array_equal(out.cpu().numpy(), np.where(orc.owner % 2 == 1, a, 0.0))
    finally:
        glm.close()
