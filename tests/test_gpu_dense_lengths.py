"""Dense rows around the lengths where the prepare kernel changes: 64 and 128 columns, one piece and more, odd lengths, with few
blocks (short-row kernel up to 128 columns) and with more than it takes at once. Against the oracle within the parity
tolerances."""
import pytest

pytestmark = pytest.mark.gpu

from parity_util import run_parity  # noqa: E402
from test_gpu_parity import tiny_dense  # noqa: E402


@pytest.mark.parametrize("loss", ["hinge", "logistic"])
@pytest.mark.parametrize("n,d,K", [(700, 63, 5), (700, 64, 5), (700, 65, 5), (700, 68, 5), (700, 100, 3), (700, 127, 5), (700, 128, 5), (24000, 64, 40),
                                   (24000, 65, 40), (24000, 68, 40), (24000, 127, 40), (24000, 128, 40), (900, 131, 4), (900, 192, 4), (900, 260, 4)])
def test_prepare_lengths(loss, n, d, K):
    run_parity(tiny_dense(n, d, seed=d, loss=loss, K=K, lam=2.0 / n), rounds=2)
