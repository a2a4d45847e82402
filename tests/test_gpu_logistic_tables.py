"""The logistic step from tables (look-ahead solver) over the range of q = sigma' |x|^2 / (lambda n): both table sizes,
their limits, and the root search beyond them, against the oracle within the parity tolerances (a table value is within
1.6e-7 of the exact step, the fp32 dot products carry 1e-6)."""
import pytest

pytestmark = pytest.mark.gpu

from parity_util import run_parity  # noqa: E402
from test_gpu_parity import tiny_csr, tiny_dense  # noqa: E402


@pytest.mark.parametrize("q", [1e-3, 0.5, 8.0, 150.0, 170.0, 5e3, 3.9e4, 3e5])
@pytest.mark.parametrize("fmt", ["dense", "csr"])
def test_step_over_q(fmt, q):
    # lambda n such that the largest coordinate's q is about the one asked for
    make = (lambda lam: tiny_dense(515, 7, seed=3, loss="logistic", K=4, lam=lam)) if fmt == "dense" else \
        (lambda lam: tiny_csr(515, 60, seed=3, loss="logistic", K=4, zero_rows=(3,)))
    w = make(1.0)
    sq = max(float((r * r).sum()) for r in (w.values.reshape(515, 7) if fmt == "dense" else
                                            [w.values[w.indptr[i]:w.indptr[i + 1]] for i in range(515)]))
    w.lam = 4.0 * sq / q / 515
    run_parity(w, rounds=3)


@pytest.mark.parametrize("q,margin", [(0.5, 4.0), (0.5, 12.0), (0.5, 24.0), (100.0, 0.0), (100.0, 14.0), (3e3, 0.0), (3.9e4, 0.0), (3.9e4, 16.0)])
def test_small_states_relative_to_themselves(q, margin):
    # every state ends between e^-margin and a few / q. A state is the sum of a few fp32 terms of 30 at most (2e-6 each way)
    # and enters the result as e^state: 1e-5 leaves room for a handful of them, whatever the size of the result
    import numpy as np
    from parity_util import make_pair, rel_l2
    n, d = 515, 7
    w = tiny_dense(n, d, seed=3, loss="logistic", K=1, lam=1.0)
    X = w.values.reshape(n, d)
    w.labels = np.where(X[:, 0] >= 0, 1.0, -1.0).astype(np.float32)
    X[:, 0] = w.labels * (1.0 + 0.1 * np.abs(X[:, 0]))
    w.lam = float(np.float32((X.astype(np.float64) ** 2).sum(1).max() / q / n))
    orc, glm = make_pair(w)
    try:
        orc.partition(1, 1)
        glm.partition(1, 1)
        v = np.zeros(d)
        v[0] = np.float32(margin * w.lam * n)
        orc.v[:] = v
        glm.set_state(orc.state.astype(np.float32), v.astype(np.float32), 0)
        orc.cocoa_round(40, 1.0)
        glm.cocoa_round(40, 1.0)
        at = orc.permutation(0, 0)[:40]
        a, b = np.abs(glm.get_alpha()[at].astype(np.float64)), np.abs(orc.state[at])
        assert (np.abs(a - b) / b).max() <= 1e-5, (np.abs(a - b) / b).max()
    finally:
        glm.close()


@pytest.mark.parametrize("fmt", ["dense", "csr"])
def test_no_memory_for_tables(fmt, monkeypatch):
    # an allocator that refuses what the tables would take (32 KB a block): the look-ahead solver runs without them
    from paper_1909_04885_b200 import binding
    w = tiny_dense(4000, 28, seed=3, loss="logistic", K=4) if fmt == "dense" else tiny_csr(4000, 60, seed=3, loss="logistic", K=4)
    serve = binding._TorchAllocator._alloc
    refused = []

    def limited(self, ctx, nbytes):
        if nbytes > (3_000_000 if fmt == "dense" else 6_000_000):
            refused.append(nbytes)
            return None
        return serve(self, ctx, nbytes)
    monkeypatch.setattr(binding._TorchAllocator, "_alloc", limited)
    run_parity(w, rounds=2)
    assert len(refused) == 1
    glm = binding.from_workload(w)
    try:
        glm.partition(4, 1)
        assert glm.cocoa_round(0, 4.0, stats=True)["solver_variant"] in (4, 5)
    finally:
        glm.close()


def long_rows_by_chunks():
    """Rows of 80 ids, 20 partitions by chunks: record slots as long as the arrays for 3 072 entries take, and tables of 32 bins beside them,
    leave little of shared memory (a process of its own: the library looks once whether it is to write a log)."""
    import numpy as np
    from paper_1909_04885_b200.datagen import Phase, Workload
    from parity_util import make_pair, rel_l2
    n, d, K = 4000, 160, 20
    rng = np.random.default_rng(5)
    ids = 2 * np.arange(80) + rng.integers(0, 2, (n, 80))
    w = Workload("long", "logistic", "csr", n, d, (rng.standard_normal(n * 80) / 9.0).astype(np.float32), np.where(rng.random(n) < 0.5, 1.0, -1.0).astype(np.float32),
                 10.0 / n, 1, [Phase(0, K, 1, float(K))], np.arange(n + 1, dtype=np.int64) * 80, ids.reshape(-1).astype(np.int32))
    orc, glm = make_pair(w)
    with glm:
        for x in (orc, glm):
            x.partition_chunks(K, 7, np.linspace(0, n, K + 1).astype(np.int64), np.arange(K, dtype=np.int32))
            x.cocoa_round(0, float(K))
        assert rel_l2(glm.get_alpha(), orc.state) <= 1e-4 and rel_l2(glm.get_v(), orc.v) <= 1e-4


def test_long_slots_leave_room_for_tables():
    import os
    import subprocess
    import sys
    here = os.path.dirname(os.path.abspath(__file__))
    root = os.path.dirname(here)
    r = subprocess.run([sys.executable, "-c", "import sys; sys.path.insert(0, %r); import test_gpu_logistic_tables as t; t.long_rows_by_chunks()" % here],
                       env=dict(os.environ, CHICLE_LOG="1", PYTHONPATH=root), cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    assert "table-bins=32 " in r.stderr, r.stderr[-1000:]
