"""Dense rows shared out over a cluster (look-ahead solver): row lengths around the slices' edges, odd lengths, many
partitions, up to the longest (3 072) and one beyond (the ring solver), against the oracle within the parity tolerances."""
import pytest

pytestmark = pytest.mark.gpu

from parity_util import run_parity  # noqa: E402
from test_gpu_parity import tiny_dense  # noqa: E402


@pytest.mark.parametrize("loss", ["hinge", "logistic"])
@pytest.mark.parametrize("d,K", [(127, 4), (128, 4), (129, 4), (255, 3), (257, 4), (385, 2), (500, 40), (769, 80), (1023, 3), (3071, 2), (3072, 2),
                                 (3073, 2)])
def test_row_lengths(loss, d, K):
    run_parity(tiny_dense(333, d, seed=d, loss=loss, K=K, lam=0.05), rounds=2)
