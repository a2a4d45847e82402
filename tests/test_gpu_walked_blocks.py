"""Blocks that are walked in place between ordinary ones (rows longer than the prepare kernel's arrays), for clusters of eight,
two and one: against the oracle within the parity tolerances; and when a block's records are missing, the round ends with the
timeout status, every warp of the cluster returns, and the handle goes on (the missing record is a host-side test aid)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1909_04885_b200 import binding  # noqa: E402
from paper_1909_04885_b200.datagen import Phase, Workload  # noqa: E402
from parity_util import make_pair, rel_l2, run_parity  # noqa: E402


def with_long_rows(n, K, loss="hinge", d=5000, seed=3):
    rng = np.random.default_rng(seed)
    lens = np.where(rng.random(n) < 0.02, 4500, 12)  # a block of 32 has a long row as often as not
    ids = [np.sort(rng.choice(d, m, replace=False)) for m in lens]
    indptr = np.zeros(n + 1, np.int64)
    indptr[1:] = np.cumsum(lens)
    vals = rng.standard_normal(int(indptr[-1])).astype(np.float32) / np.sqrt(np.repeat(lens, lens)).astype(np.float32)
    labels = np.where(rng.random(n) < 0.5, 1.0, -1.0).astype(np.float32)
    return Workload("long_rows", loss, "csr", n, d, vals, labels, 5.0 / n, 2, [Phase(0, K, seed, float(K))], indptr,
                    np.concatenate(ids).astype(np.int32))


@pytest.mark.parametrize("loss", ["hinge", "logistic"])
@pytest.mark.parametrize("n,K", [(700, 3), (3000, 20), (5000, 60)])
def test_parity(n, K, loss):
    run_parity(with_long_rows(n, K, loss), rounds=2)


@pytest.mark.parametrize("n,K", [(700, 3), (3000, 20), (5000, 60)])
def test_missing_records(n, K, monkeypatch):
    w = with_long_rows(n, K)
    orc, glm = make_pair(w)
    try:
        orc.partition(K, 3)
        glm.partition(K, 3)
        for drop in (0, 1, 2, 3, 4, 5, 6, n // K // 32):
            monkeypatch.setenv("CHICLE_TEST_DROP_RECORD", str(drop))
            with pytest.raises(binding.ChicleError) as e:
                glm.cocoa_round(0, float(K))
                glm.duality_gap()
            assert e.value.status == binding.ERR_TIMEOUT
            monkeypatch.delenv("CHICLE_TEST_DROP_RECORD")
            glm.set_state(np.zeros(n, np.float32), np.zeros(w.n_cols, np.float32), 0)
        orc.cocoa_round(0, float(K))
        glm.cocoa_round(0, float(K))
        assert rel_l2(glm.get_alpha(), orc.state) <= 1e-4 and rel_l2(glm.get_v(), orc.v) <= 1e-4
    finally:
        glm.close()
