"""Chain kernel where a block has entries beyond the part of the model in shared memory: which instance runs (its name is read from
the log), that such entries are there in every case, and the results against the oracle within the parity tolerances.

`create` numbers the ids by frequency, so what lies beyond shared memory are the rarest ids of the data. Here those are ids that a
single block of the first round has, in one to six of its rows; the frequent ids fill shared memory, each in more rows than that."""
import functools
import os
import re
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_1909_04885_b200 import binding  # noqa: E402
from paper_1909_04885_b200.datagen import Phase, Workload  # noqa: E402
from parity_util import REL_TOL, make_pair, rel_l2, run_parity  # noqa: E402

HEAD = 40  # ids that one row in four has: lists of many entries


@functools.lru_cache(maxsize=None)
def blocks_of(n, K):
    """The blocks of the first round, partition after partition."""
    orc = oracle.CocoaOracle("hinge", "csr", n, 1, np.zeros(0, np.float32), np.ones(n, np.float32), 1.0, np.zeros(n + 1, np.int64), np.zeros(0, np.int32))
    orc.partition(K, 1)
    return [orc.permutation(0, k)[i:i + 32] for k in range(K) for i in range(0, int(orc.part_off[k + 1] - orc.part_off[k]), 32)]


@functools.lru_cache(maxsize=2)
def workload(loss, K, blocks, near, times, C, longest, more, walked):
    """`near` ids in `times` rows each; then the ids of single blocks: from block to block few of them, many, some and none, per CTA.
    Blocks `walked` of the first two partitions have a row that is too long for a block's arrays."""
    rng = np.random.default_rng(1)
    n = K * blocks * 32 - 5
    m = C * more
    lists = [[1] * 4 * m + [2] * 2 * m, [1] * 20 * m + [2] * 12 * m + [min(3, longest)] * 6 * m + [longest] * 2 * m, [1] * 8 * m + [2] * 4 * m + [min(3, longest)] * 4 * m, []]
    row, ids = np.nonzero(rng.random((n, HEAD)) < 0.25)
    row, ids = [row, np.arange(near * times) % n], [ids, HEAD + rng.permutation(np.repeat(np.arange(near), times))]
    at = HEAD + near
    for b, members in enumerate(blocks_of(n, K)):
        for many in lists[b % 4]:
            if many <= len(members):
                row.append(rng.choice(members, many, replace=False))
                ids.append(np.full(many, at))
                at += 1
        if b < 2 * blocks and b % blocks in walked:
            row.append(np.full(2100, members[len(members) // 2]))
            ids.append(HEAD + rng.choice(near, 2100, replace=False))
    key = np.unique(np.concatenate(row).astype(np.int64) * at + np.concatenate(ids))
    row, ids = key // at, rng.permutation(at)[key % at]
    order = np.lexsort((ids, row))
    row, ids = row[order], ids[order]
    count = np.bincount(row, minlength=n)
    vals = (rng.standard_normal(ids.size) / np.sqrt(count[row])).astype(np.float32)
    return Workload("far", loss, "csr", n, at, vals, np.where(rng.random(n) < 0.5, 1.0, -1.0).astype(np.float32), 5.0 / n, 2,
                    [Phase(0, K, 1, float(K))], indptr=np.concatenate([[0], np.cumsum(count)]).astype(np.int64), indices=ids.astype(np.int32))


@functools.lru_cache(maxsize=2)
def uniform(loss, K, blocks, d, per):
    """Rows of `per` ids, all about equally rare."""
    rng = np.random.default_rng(3)
    n = K * blocks * 32 - 5
    ids = (np.arange(per) * (d // per) + rng.integers(0, d // per, (n, per))).reshape(-1).astype(np.int32)
    return Workload("uniform", loss, "csr", n, d, (rng.standard_normal(n * per) / np.sqrt(per)).astype(np.float32), np.where(rng.random(n) < 0.5, 1.0, -1.0).astype(np.float32),
                    5.0 / n, 2, [Phase(0, K, 1, float(K))], indptr=np.arange(n + 1, dtype=np.int64) * per, indices=ids)


def far_entries(w, K, C, on_chip):
    """Of the first round, per block and CTA: entries beyond the first `on_chip` ids by frequency, rows of the id there that most rows
    share, lists of ids that several rows share (anywhere)."""
    count = np.bincount(w.indices, minlength=w.n_cols)
    rank = np.empty(w.n_cols, np.int64)
    rank[np.lexsort((np.arange(w.n_cols), -count))] = np.arange(w.n_cols)
    out = []
    for members in blocks_of(w.n_rows, K):
        ids = np.concatenate([rank[w.indices[w.indptr[c]:w.indptr[c + 1]]] for c in members])
        u, rows = np.unique(ids, return_counts=True)
        for c in range(C):
            mine, far = u % C == c, (u % C == c) & (u >= on_chip)
            out.append((rows[far].sum(), rows[far].max(initial=0), (rows[mine] > 1).sum()))
    return np.array(out)


# name: (workload, environment, instance, CTAs, depth)
W1, W2, W4, W8 = ("hinge", 64, 12, 37_600, 7, 1, 6, 1, ()), ("hinge", 30, 60, 84_000, 7, 2, 6, 1, ()), ("hinge", 16, 48, 176_000, 4, 4, 3, 1, ()), ("hinge", 9, 120, 366_000, 3, 8, 2, 1, ())
CASES = {
    "C=1": (W1, {}, "far-warp", 1, 1),
    "C=1, two ahead": (("hinge", 64, 12, 41_000, 7, 1, 6, 1, ()), {"CHICLE_LA_DEPTH": "2"}, "cold", 1, 2),
    "C=1, tables": (("logistic", 64, 12, 26_000, 7, 1, 6, 1, ()), {}, "early", 1, 1),
    "C=1, walked": (("hinge", 64, 12, 24_900, 7, 1, 6, 1, (0, 4, 5, 7)), {}, "far-warp", 1, 1),
    "C=2": (W2, {}, "far-warp", 2, 2),
    "C=2, one ahead": (W2, {"CHICLE_LA_DEPTH": "1"}, "far-warp", 2, 1),
    "C=2, three launches": (W2, {"CHICLE_LA_SLICES": "3"}, "far-warp", 2, 2),
    "C=2, tables": (("logistic", 30, 24, 58_500, 7, 2, 6, 1, ()), {}, "cold", 2, 2),
    "C=2, no tables": (("logistic", 30, 24, 86_000, 7, 2, 6, 1, ()), {"CHICLE_LA_TABLES": "0"}, "cold", 2, 2),
    "C=2, walked": (("hinge", 30, 60, 78_000, 7, 2, 6, 1, (0, 5, 6, 9, 59)), {}, "far-warp", 2, 2),
    "C=4": (W4, {}, "far-warp", 4, 2),
    "C=8": (W8, {}, "far-warp", 8, 2),
    "C=8, one ahead": (W8, {"CHICLE_LA_DEPTH": "1"}, "far-warp", 8, 1),
    "some more, C=4": (("hinge", 16, 48, 204_000, 4, 4, 3, 1, ()), {}, "cold", 4, 2),
    "many, C=1": (("hinge", 64, 6, 36_000, 7, 1, 6, 3, ()), {}, "early", 1, 1),
    "many, C=2": (("hinge", 30, 16, 82_000, 7, 2, 6, 2, ()), {}, "cold", 2, 2),
    "many, C=2, one ahead": (("hinge", 30, 16, 82_000, 7, 2, 6, 2, ()), {"CHICLE_LA_DEPTH": "1"}, "early", 2, 1),
    "many, C=2, walked": (("hinge", 30, 16, 72_000, 7, 2, 6, 2, (0, 5, 6, 9, 15)), {}, "cold", 2, 2),
    "many, C=1, walked": (("hinge", 64, 12, 32_000, 7, 1, 6, 1, (0, 4, 5, 7)), {}, "early", 1, 1),
    "very many, C=2": (("hinge", 30, 16, 100_000, 7, 2, 6, 2, ()), {}, "cold", 2, 2),
    "most, C=2": (("hinge", 30, 48, 1_000_000, 20), {}, "early", 2, 2),
    "long, C=1": (("hinge", 40, 3, 60_000, 60), {}, "cold", 1, 1),
    "many, C=4, tables": (("logistic", 16, 48, 160_000, 4, 4, 3, 1, ()), {}, "cold", 4, 2),
}


@functools.lru_cache(maxsize=None)
def by_topic(together):
    """36 000 ids in two rows each; `together`: of the first sixth of the rows."""
    rng = np.random.default_rng(2)
    n, near, rare = 36_480, 57_000, 36_000
    row, ids = np.nonzero(rng.random((n, HEAD)) < 0.2)
    row = np.concatenate([row, np.arange(near * 7) % n, rng.integers(0, n // 6 if together else n, 2 * rare)])
    ids = np.concatenate([ids, HEAD + rng.permutation(np.repeat(np.arange(near), 7)), HEAD + near + np.arange(2 * rare) % rare])
    key = np.unique(row.astype(np.int64) * (HEAD + near + rare) + ids)
    row, ids = key // (HEAD + near + rare), key % (HEAD + near + rare)
    count = np.bincount(row, minlength=n)
    return Workload("topics", "hinge", "csr", n, HEAD + near + rare, (rng.standard_normal(ids.size) / np.sqrt(count[row])).astype(np.float32),
                    np.where(rng.random(n) < 0.5, 1.0, -1.0).astype(np.float32), 5.0 / n, 4, [Phase(0, 30, 1, 30.0)],
                    indptr=np.concatenate([[0], np.cumsum(count)]).astype(np.int64), indices=ids.astype(np.int32))


def run_chunks(w, K=30):
    orc, glm = make_pair(w)
    with glm:
        for chunks in (False, True, False, True):
            for x in (orc, glm):
                if chunks:
                    x.partition_chunks(K, 7, np.linspace(0, w.n_rows, K + 1).astype(np.int64), np.arange(K, dtype=np.int32))
                else:
                    x.partition(K, 5)
                x.cocoa_round(0, float(K))
            assert rel_l2(glm.get_alpha(), orc.state) <= REL_TOL and rel_l2(glm.get_v(), orc.v) <= REL_TOL


def run_all():
    """(a process of its own: the library looks once whether it is to write a log)"""
    for name, (args, env, *_) in CASES.items():
        os.environ.update(env)
        w = (workload if len(args) > 5 else uniform)(*args)
        print("case " + name, file=sys.stderr, flush=True)
        try:
            run_parity(w, rounds=2)
            out = []
            for _ in range(2):
                with binding.from_workload(w) as glm:
                    glm.partition(w.phases[0].K, 1)
                    glm.cocoa_round(0)
                    out.append((glm.get_alpha().copy(), glm.get_v().copy()))
            assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1]), "two runs differ"
            print("passed", file=sys.stderr, flush=True)
        except AssertionError as e:
            print("failed: %s" % e, file=sys.stderr, flush=True)
        for k in env:
            del os.environ[k]
    for together in (False, True):
        print("case %s" % together, file=sys.stderr, flush=True)
        run_chunks(by_topic(together))


@pytest.fixture(scope="module")
def logs():
    here = os.path.dirname(os.path.abspath(__file__))
    root = os.path.dirname(here)
    r = subprocess.run([sys.executable, "-c", "import sys; sys.path.insert(0, %r); import test_gpu_far_warp as t; t.run_all()" % here],
                       env=dict(os.environ, CHICLE_LOG="1", PYTHONPATH=root), cwd=root, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    parts = re.split(r"^case (.*)\n", r.stderr, flags=re.M)
    return dict(zip(parts[1::2], parts[2::2]))


@pytest.mark.parametrize("name", list(CASES))
def test_entries_beyond_shared_memory(logs, name):
    args, _, instance, C, depth = CASES[name]
    log, w = logs[name], (workload if len(args) > 5 else uniform)(*args)
    assert "\npassed" in log, log[-2000:]
    rounds = re.findall(r"round (\d+).*ctas/partition=(\d+) depth=(\d+) chain=(\S+) on-chip=(\d+) .*walked in place: (\d+)", log)
    assert [(r[1], r[2], r[3]) for r in rounds] == [(str(C), str(depth), instance)] * 4, rounds
    walked, longest = (2 * len(args[8]), args[6]) if len(args) > 5 else (0, 1)
    # (beside those, blocks that share more ids than a record slot is sized for from the ids' frequencies)
    sized = C < 8 and instance == "far-warp"
    assert walked <= int(rounds[0][5]) <= walked + (0 if sized else 0.05 * len(blocks_of(w.n_rows, args[1]))), rounds
    far, most, lists = far_entries(w, args[1], C, int(rounds[0][4])).T
    # more than the far warp keeps in registers, few and none; lists longer than it keeps, lists beyond the first 32
    assert far.max() > 64 and (far > 64).sum() >= 0.03 * far.size and (far < 24).sum() >= (0.1 * far.size if instance == "far-warp" else 0)
    assert most.max() >= longest and (instance != "far-warp" or lists.max() > 32), (far.mean(), most.max(), lists.max())


@pytest.mark.parametrize("together,instance", [(False, "far-warp"), (True, "cold")])
def test_partitions_by_chunks(logs, together, instance):
    """Rows sorted by topic: the partitions that have all the rare ids have six times the average, more than a far warp keeps up with."""
    found = re.findall(r"ctas/partition=2 .*chain=(\S+) .*walked in place: 0\n", logs[str(together)])
    assert found == ["far-warp", instance, "far-warp", instance], logs[str(together)]
