"""Partition maps and visiting orders at the sizes where the bucketed kernels change path: integer results, bit-exact
against the oracle (no tolerance)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from paper_1909_04885_b200 import binding  # noqa: E402

import oracle  # noqa: E402
from parity_util import check_partition, make_pair  # noqa: E402
from test_gpu_parity import tiny_dense  # noqa: E402
from paper_1909_04885_b200.datagen import Phase  # noqa: E402


# n / K around: one CTA's arrays (1 024, 4 096 per partition), the one-launch partition's limit (131 072 ids), 256
# partitions per pass of the member grouping, buckets of one partition
@pytest.mark.parametrize("n,K,seed", [(1024, 1, 1), (1025, 1, 2), (4096, 1, 3), (4097, 1, 4), (33, 8, 5), (131072, 16, 6), (131073, 16, 7),
                                      (140001, 256, 8), (140001, 257, 9), (131072, 513, 10), (300007, 3, 11), (600000, 70000, 12)])
def test_partition_and_orders(n, K, seed):
    w = tiny_dense(n, 1, seed=1, K=K)
    w.phases = [Phase(0, K, seed, float(K))]
    orc, glm = make_pair(w)
    try:
        orc.partition(K, seed)
        glm.partition(K, seed)
        check_partition(orc, glm, perm_rounds=(0, 5))
    finally:
        glm.close()


@pytest.mark.parametrize("n,K", [(1, 1), (31, 31), (8192, 512), (8192, 513), (131072, 3), (131072, 512), (131072, 131072), (99991, 4000)])
def test_noalloc_map(n, K):
    import torch
    orc, glm = make_pair(tiny_dense(n, 1, seed=1, K=K))
    glm.close()
    orc.partition(K, 77)
    owner = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    members = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    binding.partition_noalloc(n, K, 77, owner, members, stream=torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert np.array_equal(owner.cpu().numpy(), orc.owner)
    assert np.array_equal(members.cpu().numpy(), np.argsort(orc.owner, kind="stable"))


# rounds that walk only the head of the visiting orders (H steps, or a budget each): the state afterwards is the oracle's
@pytest.mark.parametrize("n,K,H", [(30000, 3, 1), (30000, 3, 513), (30000, 2, 14999), (30000, 4, 9000)])
def test_short_rounds(n, K, H):
    w = tiny_dense(n, 6, seed=2, K=K)
    orc, glm = make_pair(w)
    try:
        orc.partition(K, 9)
        glm.partition(K, 9)
        for r in range(2):
            orc.cocoa_round(H, float(K))
            glm.cocoa_round(H, float(K))
        steps = np.array([(k * 4001) % (n // K) for k in range(K)], np.int64)
        orc.cocoa_round(steps=steps, sigma_prime=float(K))
        glm.cocoa_round(steps=steps, sigma_prime=float(K))
        a = glm.get_alpha().astype(np.float64)
        # 32-bit dot products of 6 terms, a few thousand steps: 1e-7 relative each, 1e-5 leaves room for their sum
        assert np.linalg.norm(a - orc.state) <= 1e-5 * np.linalg.norm(orc.state)
    finally:
        glm.close()


# more than 512 partitions of given sizes: one that holds nearly all ids, a few large ones, small ones only; around the sizes
# where the one-launch kernel stops
@pytest.mark.parametrize("n,K,big", [(131072, 600, [130000]), (131072, 513, [40000, 40000, 40000]), (32768, 600, [10]), (32769, 1100, []), (2000, 600, [900]),
                                     (32768, 1024, []), (20011, 4000, [3000])])
def test_many_uneven_partitions(n, K, big):
    import time
    sizes = np.ones(K, np.int64)
    sizes[7:7 + len(big)] = big
    rest = [k for k in range(K) if not 7 <= k < 7 + len(big)]
    left = n - int(sizes.sum())
    sizes[rest] += left // len(rest)
    sizes[rest[-1]] += n - int(sizes.sum())
    orc, glm = make_pair(tiny_dense(n, 1, seed=1, K=K))
    try:
        orc.partition(K, 5, sizes)
        glm.partition(K, 5, sizes)
        check_partition(orc, glm, perm_rounds=(3,))
        took = []
        for _ in range(5):
            t = time.perf_counter()
            glm.partition(K, 6, sizes)
            took.append(time.perf_counter() - t)
        # a few launches over n ids (0.15 ms); comparing all pairs of the largest partition would be of the order of 20 ms
        assert min(took) < 5e-3, took
    finally:
        glm.close()


# visiting orders where one partition is much longer than the others (its elements are shared out over all CTAs): sizes around
# the rule's line, short and whole orders
@pytest.mark.parametrize("n,K,big", [(300007, 1300, 200000), (300007, 1300, 5000), (300007, 40, 260000), (150001, 20000, 120000), (9300, 1200, 8101)])
def test_orders_of_uneven_partitions(n, K, big):
    sizes = np.ones(K, np.int64)
    sizes[K // 2] = big
    rest = [k for k in range(K) if k != K // 2]
    sizes[rest] += (n - int(sizes.sum())) // len(rest)
    sizes[rest[-1]] += n - int(sizes.sum())
    orc, glm = make_pair(tiny_dense(n, 1, seed=1, K=K))
    try:
        orc.partition(K, 5, sizes)
        glm.partition(K, 5, sizes)
        check_partition(orc, glm, perm_rounds=(0, 7))
        H = 1 if int(sizes.min()) < 3 else 3
        for r in range(2):
            orc.cocoa_round(H, float(K))
            glm.cocoa_round(H, float(K))
        a = glm.get_alpha().astype(np.float64)
        # 32-bit products of one term, three steps a partition
        assert np.linalg.norm(a - orc.state) <= 1e-5 * np.linalg.norm(orc.state)
    finally:
        glm.close()
