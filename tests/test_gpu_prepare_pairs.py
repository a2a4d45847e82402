"""Sparse prepare kernel at the edges of its table and pair lists: ids on either side of the slots without tries, rows that are so
alike that a warp's list of entries with pairs overflows, blocks that just fit each size of the arrays and just do not, ids that collide in
the hashed slots. Against the oracle within the parity tolerances."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
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
    """All rows have the same ids: every entry has up to 31 partners in its block and 32 in the one before. Rows of 50: the arrays for 2 016
    entries; of 63 and 64: for 3 072; of 90 and more: for 4 064, which is 127 a row. (Blocks at the limits of the others: below.)"""
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


def blocks_at_the_limit(limit, more):
    """Rows of which 16 in every block are short and 16 long, with 900 ids; but two blocks of `limit` entries, `limit` / 32 ids that all their
    rows share and no others have (ids beyond the slots without tries), the first of them with `more` entries on top."""
    n, K, near = 2560, 2, 900
    short, long_ = {2016: (20, 70), 3072: (50, 110), 4064: (60, 140)}[limit]
    rng = np.random.default_rng(limit)
    orc = oracle.CocoaOracle("hinge", "csr", n, 1, np.zeros(0, np.float32), np.ones(n, np.float32), 1.0, np.zeros(n + 1, np.int64), np.zeros(0, np.int32))
    orc.partition(K, 3)
    rows = [None] * n
    for k in range(K):
        order = orc.permutation(0, k)
        for i, c in enumerate(order):
            if k == 0 and i // 32 in (1, 2):
                rows[c] = np.arange(near, near + limit // 32 + (more if i == 40 else 0))
            else:
                rows[c] = np.sort(rng.choice(near, short if i & 1 else long_, replace=False))
    return rows_of("hinge", rows, K, 3)


LIMITS = [(limit, more) for limit in (2016, 3072, 4064) for more in (0, 1)]


def run_limits():
    """(a process of its own: the library looks once whether it is to write a log)"""
    for limit, more in LIMITS:
        print("case %d %d" % (limit, more), file=sys.stderr, flush=True)
        run_parity(blocks_at_the_limit(limit, more), rounds=2)


@pytest.fixture(scope="module")
def walked():
    here = os.path.dirname(os.path.abspath(__file__))
    root = os.path.dirname(here)
    r = subprocess.run([sys.executable, "-c", "import sys; sys.path.insert(0, %r); import test_gpu_prepare_pairs as t; t.run_limits()" % here],
                       env=dict(os.environ, CHICLE_LOG="1", PYTHONPATH=root), cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    parts = re.split(r"^case (.*)\n", r.stderr, flags=re.M)
    return {name: re.findall(r"walked in place: (\d+)", log) for name, log in zip(parts[1::2], parts[2::2])}


@pytest.mark.parametrize("limit,more", LIMITS)
def test_limits_of_the_arrays(walked, limit, more):
    """In the first round the block with `limit` entries fits, with one more it is walked in place."""
    assert int(walked["%d %d" % (limit, more)][0]) == more, walked
