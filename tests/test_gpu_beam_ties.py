"""aq_beam_search on inputs with equal scores, beyond what the candidate list holds: inputs without energy in H (zero
rows and columns: every candidate of a state ties), rows of zero scale, books of few different codewords,
more states than one chunk. Exact arithmetic (see test_gpu_beam): the codes equal the oracle's search bit
for bit."""
import numpy as np
import pytest

import aq_testutil as U
import oracle
from test_gpu_beam import W_values, exact_case, run_beam

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    U.require_gpu()


@pytest.mark.parametrize("K", [1, 5, 8, 16])
@pytest.mark.parametrize("kind", ["dead inputs", "zero scales", "two codewords", "many equal", "last better"])
def test_ties(kind, K):
    layer, W_bits, H = exact_case(24, 40, 3, 8, "f16", seed=K)
    if kind == "dead inputs":
        H[8:24, :] = 0
        H[:, 8:24] = 0
        H[30, :] = 0                          # part of a group
        H[:, 30] = 0
    elif kind == "zero scales":
        layer["scales"] = np.where(np.arange(24) % 3 == 0, 0, layer["scales"]).astype(layer["scales"].dtype)
    elif kind == "two codewords":
        layer["books"][:, 2:] = layer["books"][:, :1]
        layer["books"][:, 100] = layer["books"][:, 1]
    elif kind == "many equal":
        layer["books"][1:, 40:] = layer["books"][1:, 39:40]
    else:                                     # the best codeword comes after hundreds of equal ones
        layer["books"][:, :255] = layer["books"][:, :1]
    lam = [1.0, 2.0, 1.0]
    want = oracle.beam_update(layer, W_values(W_bits, "f16"), H.astype(np.float64), lam, K)
    assert np.array_equal(run_beam(layer, W_bits, H, lam, K), want)
