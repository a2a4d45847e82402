"""What a user of the framework has it do, as measurable cases.

A program that trains with this library creates a problem, partitions its coordinates, and then repeats one step: a
CoCoA round (K local solvers, their updates added) and the duality gap, reading the model back. The cases cover that
step over the losses, formats and sizes of the repository's configurations and between them, the elastic schedule
(a repartition between rounds), rounds of a given number of steps, partitions of unequal sizes with a step budget each,
a whole job that starts from host arrays, and the partition map without allocation.

All inputs are synthetic and drawn from the seed on the GPU.
"""
import math

import numpy as np
import torch

from paper_1909_04885_b200 import binding

DEV = "cuda"


# ------------------------------------------------------------------------------------------------ cases
def _train(name, loss, fmt, n, d, K, per=0.0, zipf=0.0, lam_n=10.0, H=0):
    """A training step on n coordinates: rows of length `d` (dense), rows with `per` of d ids each (CSR), columns
    with `per` of d rows each (CSC, ridge). per: mean entries per coordinate (Poisson), or exact if `fixed`."""
    return {"name": name, "kind": "train", "loss": loss, "fmt": fmt, "n": n, "d": d, "K": K, "per": per, "fixed": False,
            "zipf": zipf, "lam_n": lam_n, "H": H}


def listed():
    return [
        # the partition map where nothing may be allocated (a pool frozen at start-up): the smallest call there is
        {"name": "map_noalloc", "kind": "map", "n": 20_000, "K": 16},
        # an interactive fit on a small dense table: launches and latency
        _train("dense_small", "hinge", "dense", 10_000, 100, 4, lam_n=1.0),
        # dense rows longer than the short-row kernels take
        _train("dense_wide", "hinge", "dense", 100_000, 500, 16),
        # the tall dense table with a logistic loss, the largest dense configuration
        _train("dense_tall_logistic", "logistic", "dense", 11_000_000, 28, 32, lam_n=11.0),
        # bag-of-words-like sparse rows: the mid-size configuration, one local epoch per round
        _train("csr", "hinge", "csr", 1_000_000, 100_000, 16, per=50.0, zipf=1.1),
        # the same data with short rounds (communication after a thirty-second of an epoch)
        _train("csr_short_rounds", "hinge", "csr", 1_000_000, 100_000, 16, per=50.0, zipf=1.1, H=2_000),
        # hashed rows of exactly 39 ids: the largest configuration, in its long phase
        dict(_train("hashed_large", "hinge", "csr", 45_000_000, 1_000_000, 16, per=39.0, zipf=1.05, lam_n=4.5), fixed=True),
        # the elastic schedule at an eighth of that size: scale out, a round, scale in, a round, the gap
        {"name": "hashed_elastic", "kind": "elastic", "loss": "hinge", "fmt": "csr", "n": 5_625_000, "d": 125_000, "K": 64, "K2": 16,
         "per": 39.0, "fixed": True, "zipf": 1.05, "lam_n": 4.5, "H": 0},
        # ridge over feature partitions: uniform row ids, many partitions
        _train("ridge", "ridge", "csc", 2_000_000, 350_000, 128, per=81.0, lam_n=100.0),
        # slow and fast tasks: ragged partition sizes and a step budget for each, logistic loss on sparse rows
        {"name": "budgets_logistic", "kind": "budgets", "loss": "logistic", "fmt": "csr", "n": 300_007, "d": 30_011, "K": 11,
         "per": 20.0, "fixed": False, "zipf": 1.05, "lam_n": 10.0, "H": 0},
        # a whole job from pinned host arrays: create, partition, one round, gap, the model back on the host
        {"name": "job_from_host", "kind": "job", "loss": "hinge", "fmt": "csr", "n": 1_000_000, "d": 100_000, "K": 16, "per": 50.0,
         "fixed": False, "zipf": 1.1, "lam_n": 10.0, "H": 0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["map", "dense", "dense", "wide", "csr", "csr", "hashed", "elastic", "ridge", "budgets", "job"])
    if kind == "map":
        n = _log(rng, 500, 131_072)
        return {"kind": "map", "n": n, "K": min(n, _log(rng, 2, 300))}
    if kind in ("dense", "wide"):
        loss = rng.choice(["hinge", "logistic"])
        d = rng.randint(4, 128) if kind == "dense" else _log(rng, 129, 2_000)
        n = _log(rng, 2_000, min(4_000_000, 250_000_000 // d)) if kind == "dense" else _log(rng, 2_000, 100_000_000 // d)
        c = _train("", loss, "dense", n, d, _log(rng, 2, 64))
    elif kind == "ridge":
        c = _train("", "ridge", "csc", _log(rng, 20_000, 2_000_000), _log(rng, 5_000, 350_000), _log(rng, 4, 128),
                   per=float(rng.randint(10, 90)), lam_n=100.0)
    else:
        n = _log(rng, 10_000, 4_000_000) if kind in ("csr", "hashed") else _log(rng, 10_000, 1_000_000)
        c = _train("", rng.choice(["hinge", "hinge", "logistic"]), "csr", n, _log(rng, 3_000, 300_000), _log(rng, 2, 64),
                   per=float(rng.randint(8, 80)), zipf=rng.choice([1.05, 1.1, 1.2]))
        if kind == "hashed":
            c["fixed"], c["per"] = True, float(rng.choice([26, 39, 39, 64]))
        elif kind in ("elastic", "budgets", "job"):
            c["kind"] = kind
        if kind == "elastic":
            c["K2"] = max(2, c["K"] // rng.choice([2, 4]))
    # a partition's walk is sequential: none longer than the largest listed cases' walks take
    c["n"] = min(c["n"], c["K"] * (60_000 if kind == "wide" else 150_000 if c["loss"] == "logistic" else 300_000))
    if c["kind"] == "train" and rng.random() < 0.3:  # rounds that are not one local epoch long
        c["H"] = max(1, int(c["n"] / c["K"] * rng.choice([0.02, 0.1, 0.4, 1.5])))
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------------ inputs
def _ids(n, d, per, fixed, zipf, g):
    """For n coordinates, distinct ids of [0, d): Poisson(per) of them (exactly `per` if fixed), Zipf-distributed under
    a random numbering, or uniform where zipf is 0. Ascending inside a coordinate. Drawn rank after rank: the next
    rank is the smallest of the draws that are left, given that it lies beyond the last one."""
    if fixed:
        counts = torch.full((n,), int(per), dtype=torch.int64, device=DEV)
    else:
        counts = torch.poisson(torch.full((n,), per, dtype=torch.float64, device=DEV), generator=g).to(torch.int64)
    counts.clamp_(1, d)
    indptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(counts, 0, out=indptr[1:])
    out = torch.empty(int(indptr[-1]), dtype=torch.int32, device=DEV)
    number = torch.randperm(d, generator=g, device=DEV).to(torch.int32) if zipf else None
    p = 1.0 - zipf
    end = float(d + 1) ** p
    chunk = 1 << 21
    for r0 in range(0, n, chunk):
        cnt = counts[r0:r0 + chunk].double()
        width = int(cnt.max())
        rows = torch.full((width, cnt.numel()), d, dtype=torch.int32, device=DEV)
        last = torch.full_like(cnt, -1.0)
        above = torch.ones_like(cnt)  # share of the distribution beyond the last rank
        for j in range(width):
            left = (cnt - j).clamp_(min=1.0)
            at = above * torch.rand(cnt.shape, generator=g, dtype=torch.float64, device=DEV).pow_(1.0 / left)
            rank = (end + at * (1.0 - end)).pow_(1.0 / p).floor_().sub_(1.0)
            rank = torch.minimum(torch.maximum(rank, last + 1.0), d - left)
            last = rank
            above = (((rank + 2.0).pow_(p) - end) / (1.0 - end)).clamp_(min=0.0)
            rows[j] = rank.to(torch.int32) if fixed else torch.where(j < cnt, rank, float(d)).to(torch.int32)
        ids = rows.t().contiguous()
        if zipf:
            ids = torch.where(ids < d, number[ids.clamp(max=d - 1).long()], ids)
            ids = torch.sort(ids, dim=1).values
        out[int(indptr[r0]):int(indptr[min(n, r0 + chunk)])] = ids.reshape(-1) if fixed else ids[ids < d]
    return indptr, out


def _per_coordinate(indptr, per_entry, chunk=1 << 20):
    """Sums of consecutive runs of entries; per_entry(a, b) gives the entries a .. b - 1."""
    n = indptr.numel() - 1
    out = torch.empty(n, dtype=torch.float64, device=DEV)
    for r0 in range(0, n, chunk):
        r1 = min(n, r0 + chunk)
        a, b = int(indptr[r0]), int(indptr[r1])
        run = torch.zeros(b - a + 1, dtype=torch.float64, device=DEV)
        torch.cumsum(per_entry(a, b), 0, out=run[1:])
        at = indptr[r0:r1 + 1] - a
        out[r0:r1] = run[at[1:]] - run[at[:-1]]
    return out


def _inputs(case, seed):
    """values, labels, indptr, indices on the GPU, and n_rows, n_cols, lambda."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    n, d = case["n"], case["d"]
    kw = dict(generator=g, device=DEV)
    if case["fmt"] == "dense":
        X = torch.randn((n, d), **kw)
        score = (X @ torch.randn(d, **kw)).double() / math.sqrt(d)
        noise = 0.1 * torch.randn(n, dtype=torch.float64, **kw)
        if case["loss"] == "logistic":
            y = torch.where(torch.rand(n, dtype=torch.float64, **kw) < torch.sigmoid(3.0 * score), 1.0, -1.0)
        else:
            y = torch.where(score + noise >= 0, 1.0, -1.0)
        return X.reshape(-1), y.float(), None, None, n, d, case["lam_n"] / n
    indptr, ids = _ids(n, d, case["per"], case["fixed"], case["zipf"], g)
    counts = indptr[1:] - indptr[:-1]
    if case["fmt"] == "csc":  # n columns over d rows: values U(0, 1] scaled to rows of about unit norm
        vals = (1.0 - torch.rand(ids.numel(), **kw)) * math.sqrt(3.0 * d / (n * case["per"]))
        w = torch.randn(n, **kw) * (torch.rand(n, **kw) < 0.01)
        y = 0.01 * torch.randn(d, **kw)
        y.index_add_(0, ids, vals * torch.repeat_interleave(w, counts))
        return vals, y, indptr, ids, d, n, case["lam_n"] / d / d
    vals = torch.repeat_interleave(counts.double().rsqrt().float(), counts)
    w = torch.randn(d, **kw) * (torch.rand(d, **kw) < 0.05)
    score = _per_coordinate(indptr, lambda a, b: (vals[a:b] * w[ids[a:b]]).double())
    y = torch.where(score + 0.1 * torch.randn(n, dtype=torch.float64, **kw) > score[: 1 << 20].median(), 1.0, -1.0)
    return vals, y.float(), indptr, ids, n, d, case["lam_n"] / n


def prepare(case, seed):
    s = dict(case)
    if case["kind"] == "map":
        s["seed"] = seed
        s["owner"] = torch.empty(case["n"], dtype=torch.int32, device=DEV)
        s["members"] = torch.empty(case["n"], dtype=torch.int32, device=DEV)
        s["stream"] = torch.cuda.current_stream().cuda_stream
        return s
    values, labels, indptr, indices, n_rows, n_cols, lam = _inputs(case, seed)
    s["seed"], s["n_rows"], s["n_cols"], s["lam"] = seed, n_rows, n_cols, lam
    if case["kind"] == "job":  # pinned host arrays, and pinned memory for what comes back
        pin = lambda t: t.cpu().pin_memory().numpy()  # noqa: E731
        s["host"] = [pin(values), pin(labels), pin(indptr), pin(indices)]
        s["alpha"] = torch.empty(case["n"], dtype=torch.float32).pin_memory().numpy()
        s["v"] = torch.empty(case["d"], dtype=torch.float32).pin_memory().numpy()
        return s
    glm = binding.Glm(case["loss"], case["fmt"], n_rows, n_cols, values, labels, lam, indptr, indices)
    del values, labels, indptr, indices
    torch.cuda.empty_cache()
    K = case["K"]
    if case["kind"] == "budgets":  # partition k holds a share that grows with k; half of them may not finish theirs
        share = np.arange(2, K + 2, dtype=np.float64)
        sizes = np.maximum(1, np.floor(case["n"] * share / share.sum())).astype(np.int64)
        sizes[-1] += case["n"] - sizes.sum()
        glm.partition(K, seed, sizes)
        s["steps"] = np.where(np.arange(K) % 2 == 0, sizes, sizes * 3 // 4).astype(np.int64)
    else:
        glm.partition(K, seed)
    s["glm"] = glm
    s["alpha"] = torch.empty(case["n"], dtype=torch.float32, device=DEV)
    s["v"] = torch.empty(case["d"], dtype=torch.float32, device=DEV)
    return s


# ------------------------------------------------------------------------------------------------ a pass
def run(s):
    if s["kind"] == "map":
        binding.partition_noalloc(s["n"], s["K"], s["seed"], s["owner"], s["members"], stream=s["stream"])
        return s["owner"], s["members"]
    if s["kind"] == "job":
        values, labels, indptr, indices = s["host"]
        with binding.Glm(s["loss"], s["fmt"], s["n_rows"], s["n_cols"], values, labels, s["lam"], indptr, indices) as glm:
            glm.partition(s["K"], s["seed"])
            glm.cocoa_round(s["H"])
            gap = glm.duality_gap()
            return gap, glm.get_alpha(s["alpha"]), glm.get_v(s["v"])
    glm = s["glm"]
    if s["kind"] == "elastic":
        glm.partition(s["K"], s["seed"])
        glm.cocoa_round(s["H"])
        glm.partition(s["K2"], s["seed"] + 1)
        glm.cocoa_round(s["H"])
    elif s["kind"] == "budgets":
        glm.cocoa_round(steps=s["steps"])
    else:
        glm.cocoa_round(s["H"])
    gap = glm.duality_gap()
    return gap, glm.get_alpha(s["alpha"]), glm.get_v(s["v"])


# ------------------------------------------------------------------------------------------------ what it needs
def work(case):
    n, K = case["n"], case["K"]
    if case["kind"] == "map":
        return {"bytes": 8 * n, "flops": 0}
    d = case["d"]
    nnz = n * d if case["fmt"] == "dense" else n * case["per"]
    matrix = nnz * 4 if case["fmt"] == "dense" else nnz * 8 + n * 8
    share = min(1.0, case["H"] * K / n) if case["H"] else 1.0  # of the coordinates that a round visits
    again = max(1.0, case["H"] * K / n) if case["H"] else 1.0
    rounds = 2 if case["kind"] == "elastic" else 1
    # a round reads its coordinates' entries, labels and norms and rewrites their state; the gap, which needs the
    # round's result, reads the matrix, the labels and the state; the state and the shared vector come back
    one = share * (matrix + 16 * n) + 8 * d
    gap = matrix + 8 * n + 4 * d
    back = 8 * (n + d)
    arriving = matrix + 4 * n if case["kind"] == "job" else 0  # written where the job's arrays are put
    return {"bytes": rounds * one + gap + back + arriving, "flops": (4 * rounds * share * again + 2) * nnz}


def tolerance(case):
    if case["kind"] == "map":
        return "exact"
    # 32-bit dot products and updates in another order; the gap is a difference of two sums that are larger than it
    return {"rel": 1e-5, "max": 1e-3}
