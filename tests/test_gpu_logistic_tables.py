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
