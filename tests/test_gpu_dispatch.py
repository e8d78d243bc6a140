"""Edges of the launch and layout rules (run with -m gpu on a B200): the sizes at which a rule switches, remainders, the
smallest and largest nets of a rule's range, each against the float64 oracle."""
import numpy as np
import pytest

from parity_util import ragged_net
from test_gpu_parity import BWD_MODES, infer_parity, sdnn, torch_cuda, train_parity  # noqa: F401

pytestmark = pytest.mark.gpu


def vectors(rng, count, n):
    return rng.uniform(0, 1.0, size=(count, n)).astype(np.float32)


@pytest.mark.parametrize("n", [1023, 1024, 1041, 2100])
@pytest.mark.parametrize("B", [2, 20])
def test_ragged_rows_stored_by_length(torch_cuda, n, B):  # noqa: F811
    """Rows are sorted by length in blocks of 1024: a block short by one row, a whole one, a second block of one slice and
    one row, a third of a few slices; weights and biases keep the caller's order."""
    rng = np.random.default_rng(n + B)
    arrays = ragged_net(rng, n=n, layers=3, kmax=40, scale=0.3)
    train_parity(torch_cuda, arrays, [(vectors(rng, B, n), vectors(rng, B, n)) for _ in range(2)], eta=0.02, update_bias=True,
                 activation="sigmoid", expect_live=True)
    infer_parity(torch_cuda, arrays, vectors(rng, 3 * B, n), 2 * B, expect_nonempty=True)
