"""aq_beam_search where its candidate pruning changes form: zero prefix weights (every codeword of a
state ties), books of equal codewords and zero weights (more ties than the candidate list holds,
magnitudes below the estimates' range), one and two chunks of eight states, beams that are no power
of two. Exact arithmetic (see test_gpu_beam): the codes equal the oracle's search bit for bit."""
import numpy as np
import pytest

import aq_testutil as U
import oracle
from test_gpu_beam import W_values, exact_case, run_beam

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    U.require_gpu()


@pytest.mark.parametrize("K", [1, 3, 8, 11, 16])
@pytest.mark.parametrize("lam", [[1.0, 2.0, 1.0], [0.0, 0.0, 1.0], [1.0, 0.0, 2.0], [0.0, 0.0, 0.0]])
def test_prefix_weights_and_beams(K, lam):
    layer, W_bits, H = exact_case(24, 32, 3, 8, "f16", seed=K)
    want = oracle.beam_update(layer, W_values(W_bits, "f16"), H.astype(np.float64), lam, K)
    assert np.array_equal(run_beam(layer, W_bits, H, lam, K), want)


@pytest.mark.parametrize("B", [4, 8])
def test_ties_beyond_the_list(B):
    """Equal codewords in a book, a zero row with zero scale contributions: all candidates tie."""
    layer, W_bits, H = exact_case(16, 32, 2, B, "f16", seed=5)
    layer["books"][0][:] = layer["books"][0][0]
    layer["books"][1][:] = 0
    W_bits = W_bits.copy()
    W_bits[3] = 0
    want = oracle.beam_update(layer, W_values(W_bits, "f16"), H.astype(np.float64), [1.0, 1.0], 8)
    assert np.array_equal(run_beam(layer, W_bits, H, None, 8), want)
