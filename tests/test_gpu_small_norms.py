"""Sparse rows whose squared norms are near the smallest fp32 numbers, and below the smallest normal one: multiplying X by c and
lambda by c^2 leaves alpha as it is, so the look-ahead solver's Gram entries (most of them on ids that it does not keep in its
dense tiles) matter as much as at any other scale. Against the oracle within the parity tolerances; the norms stop where
1 / |x|^2 is still an fp32 number."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from parity_util import run_parity  # noqa: E402
from test_gpu_record_slots import sparse  # noqa: E402


@pytest.mark.parametrize("loss", ["hinge", "logistic"])
@pytest.mark.parametrize("shift", [0, 40, 59, 61, 63])
def test_scaled_rows(loss, shift):
    w = sparse(loss, 96, 90, 20, 1, 0.0, seed=5)
    w.values = np.ldexp(w.values, -shift)
    w.lam = float(np.ldexp(np.float32(0.03), -2 * shift))
    run_parity(w, rounds=3)
