"""Chain kernel where the model is longer than its part in shared memory. `create` numbers the ids by frequency, and these rows have fewer
ids than shared memory holds in most cases: what lies beyond it are ids that no row has, in the others rare ones that a block rarely
shares. Every cluster size and both depths, rounds in several launches, blocks walked in place between others, long records. Against the
oracle within the parity tolerances, and the same bits in two runs. (Entries beyond shared memory in every block: test_gpu_far_warp.py.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1909_04885_b200 import binding  # noqa: E402
from parity_util import run_parity  # noqa: E402
from paper_1909_04885_b200.datagen import Phase, Workload  # noqa: E402


def rows(loss, n, d, per, K, far, seed):
    """`per` ids a row: most of them Zipf-distributed, a share `far` of them from a few hundred of the last nine tenths of the numbers."""
    rng = np.random.default_rng(seed)
    ids = []
    for i in range(n):
        m = int(rng.binomial(per, far))
        r = set((d // 10 + (rng.integers(0, 40, m) * 9973 + rng.integers(0, 2, m) * (i % 7) * 31) % (d - d // 10)).tolist())
        while len(r) < per:
            r.add(int(min(d - 1, d ** rng.random() - 1)))
        ids.append(np.sort(np.fromiter(r, np.int32)))
    vals = (rng.standard_normal(n * per) / np.sqrt(per)).astype(np.float32)
    return Workload("far", loss, "csr", n, d, vals, np.where(rng.random(n) < 0.5, 1.0, -1.0).astype(np.float32), 5.0 / n, 2,
                    [Phase(0, K, seed, float(K))], indptr=np.arange(n + 1, dtype=np.int64) * per, indices=np.concatenate(ids).astype(np.int32))


@pytest.mark.parametrize("loss,n,d,per,K,far", [
    ("hinge", 1500, 400_000, 20, 1, 0.3), ("hinge", 2100, 300_001, 39, 9, 0.1), ("hinge", 3000, 200_000, 39, 16, 0.5), ("logistic", 2500, 400_000, 20, 30, 0.2),
    ("hinge", 4000, 120_000, 39, 64, 0.02), ("logistic", 3000, 150_000, 33, 64, 0.9), ("hinge", 2500, 100_000, 100, 70, 0.3), ("hinge", 2500, 100_000, 125, 70, 0.3)])
def test_ids_beyond_shared_memory(loss, n, d, per, K, far):
    run_parity(rows(loss, n, d, per, K, far, seed=n + K), rounds=2)


@pytest.mark.parametrize("cluster,depth", [("1", "1"), ("1", "2"), ("2", "2"), ("4", "1"), ("8", "2")])
def test_same_bits_and_slices(cluster, depth, monkeypatch):
    monkeypatch.setenv("CHICLE_LA_CLUSTER", cluster)
    monkeypatch.setenv("CHICLE_LA_DEPTH", depth)
    monkeypatch.setenv("CHICLE_LA_SLICES", "3")
    w = rows("hinge", 3000, 500_000, 30, 5, 0.3, seed=4)
    run_parity(w, rounds=2)
    out = []
    for _ in range(2):
        with binding.from_workload(w) as glm:
            glm.partition(5, 1)
            glm.cocoa_round(0)
            out.append((glm.get_alpha().copy(), glm.get_v().copy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("K", [3, 60])
def test_walked_blocks_between(K):
    """Rows of which one in 200 is longer than a block's arrays: its block is walked in place, against ids here and there."""
    w = rows("hinge", 900, 200_000, 30, K, 0.3, seed=6)
    rng = np.random.default_rng(1)
    lists = [w.indices[30 * i:30 * i + 30] for i in range(900)]
    for i in range(100, 900, 200):
        lists[i] = np.sort(rng.choice(200_000, 5000, replace=False)).astype(np.int32)
    w.indptr = np.concatenate([[0], np.cumsum([len(r) for r in lists])]).astype(np.int64)
    w.indices = np.concatenate(lists)
    w.values = np.concatenate([rng.standard_normal(len(r)) / np.sqrt(len(r)) for r in lists]).astype(np.float32)
    run_parity(w, rounds=2)
