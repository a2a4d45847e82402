"""The look-ahead solver's records find room (a block without is walked in place, some twenty times slower): rows that share most of
their ids, partitions by chunks of data sorted by topic or by length, where whole partitions differ from the average. The number
of blocks walked in place is read from the log; the results are compared with the oracle within the parity tolerances."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1909_04885_b200.datagen import Phase, Workload  # noqa: E402
from parity_util import make_pair, rel_l2  # noqa: E402


def workload(kind, n, K, seed=3):
    rng = np.random.default_rng(seed)
    if kind == "topics":  # 20 topics, sorted; 50 of a topic's 100 ids in a row
        t = np.sort(rng.integers(0, 20, n))
        ids = t[:, None] * 100 + 2 * np.arange(50) + rng.integers(0, 2, (n, 50))
        lens, d, ids = np.full(n, 50), 2000, ids.reshape(-1)
    elif kind == "lengths":  # sorted by length, few ids shared
        lens = np.sort(np.maximum(1, rng.poisson(45, n)))
        j = np.concatenate([np.arange(m) for m in lens])
        ids, d = j * 400 + rng.integers(0, 400, j.size), 400 * (int(lens.max()) + 1)
    else:  # 50 of the same 100 ids in every row
        ids = (2 * np.arange(50) + rng.integers(0, 2, (n, 50))).reshape(-1)
        lens, d = np.full(n, 50), 100
    indptr = np.zeros(n + 1, np.int64)
    indptr[1:] = np.cumsum(lens)
    vals = np.repeat(1.0 / np.sqrt(lens), lens).astype(np.float32)
    labels = np.where(rng.random(n) < 0.5, 1.0, -1.0).astype(np.float32)
    return Workload(kind, "hinge", "csr", n, d, vals, labels, 10.0 / n, 2, [Phase(0, K, seed, float(K))], indptr, ids.astype(np.int32))


def placement(n, K):
    return np.linspace(0, n, K + 1).astype(np.int64), np.arange(K, dtype=np.int32)


def logged_walks(kind, n, K, chunks):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = ("import sys; sys.path.insert(0, %r)\n"
            "from test_gpu_record_room import workload, placement\n"
            "from paper_1909_04885_b200 import binding\n"
            "glm = binding.from_workload(workload(%r, %d, %d))\n"
            "glm.partition_chunks(%d, 7, *placement(%d, %d)) if %r else glm.partition(%d, 7)\n"
            "glm.cocoa_round(0)\n" % (os.path.join(root, "tests"), kind, n, K, K, n, K, chunks, K))
    out = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, CHICLE_LOG="1", PYTHONPATH=root), cwd=root, capture_output=True, text=True,
                         timeout=300)
    assert out.returncode == 0, out.stderr[-2000:]
    m = re.findall(r"solver=(\d+).*blocks walked in place: (\d+)", out.stderr)
    assert len(m) == 1 and m[0][0] == "4", out.stderr[-2000:]
    return int(m[0][1])


@pytest.mark.parametrize("kind,n,K,chunks", [("topics", 40000, 8, True), ("topics", 40000, 64, True), ("lengths", 100000, 16, True),
                                             ("lengths", 100000, 64, True), ("alike", 60000, 8, False), ("alike", 1024000, 128, False)])
def test_no_block_is_walked_in_place(kind, n, K, chunks):
    assert logged_walks(kind, n, K, chunks) == 0


@pytest.mark.parametrize("kind", ["topics", "lengths"])
@pytest.mark.parametrize("loss", ["hinge", "logistic"])
def test_random_and_chunk_partitions_in_turn(kind, loss):
    n, K = 6000, 12
    w = workload(kind, n, K)
    w.loss = loss
    off, task = placement(n, K)
    orc, glm = make_pair(w)
    try:
        for chunks in (False, True, True, False):
            for x in (orc, glm):
                if chunks:
                    x.partition_chunks(K, 7, off, task)
                else:
                    x.partition(K, 5)
            assert np.array_equal(glm.get_partition(), orc.owner)
            orc.cocoa_round(0, float(K))
            glm.cocoa_round(0, float(K))
            assert rel_l2(glm.get_alpha(), orc.state) <= 1e-4 and rel_l2(glm.get_v(), orc.v) <= 1e-4
    finally:
        glm.close()
