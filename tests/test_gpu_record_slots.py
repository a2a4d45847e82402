"""Sparse look-ahead solver where a block's records are long or the ids flat: rows of 80 entries over many partitions (three
slots per record, no room beside the tables), few ids that every block shares, flat ids with a cluster per partition and with
more clusters than run at a time, partitions whose numbers are no multiple of what the aggregation takes at once; and more
partitions than the arguments of one kernel hold step budgets for. Against the oracle within the parity tolerances."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from parity_util import run_parity  # noqa: E402
from paper_1909_04885_b200.datagen import Phase, Workload  # noqa: E402


def sparse(loss, n, d, per, K, skew, seed):
    """n coordinates of `per` distinct ids of [0, d); the larger `skew`, the more of them on the first ids."""
    rng = np.random.default_rng(seed)
    p = (np.arange(d) + 1.0) ** -skew
    p /= p.sum()
    ids = np.concatenate([np.sort(rng.choice(d, per, replace=False, p=p)) for _ in range(n)]).astype(np.int32)
    vals = rng.standard_normal(n * per).astype(np.float32) / np.float32(np.sqrt(per))
    ridge = loss == "ridge"
    labels = rng.standard_normal(d) if ridge else np.where(rng.random(n) < 0.5, 1.0, -1.0)
    rows, cols = (d, n) if ridge else (n, d)
    return Workload("sparse", loss, "csc" if ridge else "csr", rows, cols, vals, labels.astype(np.float32), 0.05 if ridge else 5.0 / n, 2,
                    [Phase(0, K, seed, float(K))], indptr=np.arange(n + 1, dtype=np.int64) * per, indices=ids)


@pytest.mark.parametrize("loss,n,d,per,K,skew", [
    ("logistic", 4000, 3000, 80, 48, 1.2), ("hinge", 4000, 400, 80, 48, 0.0), ("hinge", 3000, 90, 80, 40, 1.0), ("logistic", 3000, 90, 80, 9, 1.0),
    ("hinge", 2500, 60000, 64, 11, 0.3), ("ridge", 3000, 5000, 60, 21, 0.0), ("ridge", 2000, 300000, 40, 128, 0.0), ("hinge", 3000, 3, 2, 7, 0.0)])
def test_records(loss, n, d, per, K, skew):
    run_parity(sparse(loss, n, d, per, K, skew, seed=n + d + K), rounds=2)


@pytest.mark.parametrize("K", [480, 481, 1300])
def test_budgets_of_many_partitions(K):
    w = sparse("hinge", 6000, 500, 5, K, 0.5, seed=K)
    run_parity(w, rounds=2, steps=lambda r: np.array([(k + r) % 4 for k in range(K)], np.int64))
