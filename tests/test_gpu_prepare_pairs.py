"""Sparse prepare kernel at the edges of its table and pair lists: ids on either side of the slots without tries, rows that are so
alike that a warp's list of entries with pairs overflows, blocks that just fit the arrays and just do not, ids that collide in
the hashed slots. Against the oracle within the parity tolerances."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from parity_util import run_parity  # noqa: E402
from paper_1909_04885_b200.datagen import Phase, Workload  # noqa: E402


def rows_of(loss, ids, K, seed):
    """Rows with the given ids each (ascending)."""
    rng = np.random.default_rng(seed)
    n, d = len(ids), 1 + max(int(r[-1]) for r in ids)
    indptr = np.concatenate([[0], np.cumsum([len(r) for r in ids])]).astype(np.int64)
    vals = np.concatenate([rng.standard_normal(len(r)) / np.sqrt(len(r)) for r in ids]).astype(np.float32)
    return Workload("pairs", loss, "csr", n, d, vals, np.where(rng.random(n) < 0.5, 1.0, -1.0).astype(np.float32), 5.0 / n, 2,
                    [Phase(0, K, seed, float(K))], indptr=indptr, indices=np.concatenate(ids).astype(np.int32))


@pytest.mark.parametrize("loss", ["hinge", "logistic"])
@pytest.mark.parametrize("d", [31, 33, 767, 768, 769, 1025, 2900])
def test_table_edges(loss, d):
    """Every id about equally frequent: ids below and above 768 meet in every block."""
    rng = np.random.default_rng(d)
    per = min(d, 40)
    run_parity(rows_of(loss, [np.sort(rng.choice(d, per, replace=False)) for _ in range(700)], 3, d), rounds=2)


@pytest.mark.parametrize("per,K", [(50, 2), (63, 5), (64, 2), (90, 2), (126, 2), (127, 2), (128, 2)])
def test_alike(per, K):
    """All rows have the same ids: every entry has up to 31 partners in its block and 32 in the one before; blocks of up to 2 016, 3 072
    and 4 064 entries are what the three sizes of arrays hold."""
    run_parity(rows_of("hinge", [np.arange(per)] * 500, K, per), rounds=2)


@pytest.mark.parametrize("per", [45, 75, 120])
def test_all_different(per):
    """No two rows share an id: as many ids in the table as there are entries."""
    run_parity(rows_of("hinge", [np.arange(i * per, (i + 1) * per) for i in range(300)], 2, per), rounds=2)


@pytest.mark.parametrize("mix", [(1, 200), (200, 1), (0, 60)])
def test_uneven_rows(mix):
    """Long and short (or empty) rows in one block."""
    rng = np.random.default_rng(7)
    ids = [np.sort(rng.choice(1500, max(1, mix[i & 1]), replace=False)) for i in range(400)]
    run_parity(rows_of("logistic", ids, 4, 3), rounds=2)
