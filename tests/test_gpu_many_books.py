"""9..16 tokens with five to eight 8-bit books (gemm_ts with eight or four copies of each book, or two
token tiles of gemv_cw), and gemv_cw over several passes of a CTA's row blocks: ragged rows and slices, warps without a unit, two, three and four passes;
y = x W_m^T of Sec. 2.2 with the prefix reconstruction of Sec. 3.2 / Sec. 5.

Tolerance: a decoded weight may be rounded once to fp16 (2^-11 of its sum of |C_k|), the rest are fp32
sums (below 2^-13 of A = |s| sum_i |x_i| sum_k |C_k|_i, as derived in test_gpu_cw)."""
import numpy as np
import pytest

import aq_testutil as U
import oracle
import paper_2606_12876_gb300 as aq
import workloads
from paper_2606_12876_gb300.linear import AQLinear, x_to_device
from test_gpu_cw import _widen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    U.require_gpu()


@pytest.mark.parametrize("out,inp,M,B,bdt,xdt,ms,tokens", [
    (4099, 4104, 8, 8, "f16", "bf16", (5, 6, 7, 8), (9, 16)),
    (700, 2312, 8, 8, "bf16", "bf16", (5, 6, 7, 8), (13,)),
    (96, 9000, 6, 8, "bf16", "f16", (5, 6), (16,)),
    (10001, 264, 2, 8, "f16", "bf16", (1, 2), (5, 8)),       # three passes, warps without a unit
    (14600, 1032, 4, 8, "f16", "f16", (1, 3, 4), (3, 8)),    # four passes, several units a warp
    (5000, 1000, 4, 4, "bf16", "f16", (4,), (2, 4, 16)),     # two passes (a token tile has half the SMs)
])
def test_books_and_passes(out, inp, M, B, bdt, xdt, ms, tokens):
    layer = workloads.make_layer(out, inp, G=8, M=M, B=B, book_dtype=bdt, book_std=0.05,
                                 scale_dtype=bdt, seed=out + M)
    x_bits = workloads.make_x(16, inp, xdt, seed=inp)
    lin = AQLinear.from_layer(layer)
    x = x_to_device(x_bits, xdt)
    absl = dict(layer, books=np.asarray(layer["books"], np.uint16) & 0x7fff,
                scales=np.asarray(layer["scales"], np.uint16) & 0x7fff)
    X = np.abs(_widen(x_bits, xdt))
    for m in ms:
        ref = oracle.product_exact(layer, x_bits, xdt, m)
        bound = (2.0 ** -11 + 2.0 ** -13) * (X @ np.abs(oracle.reconstruct_exact(absl, m)).T)
        for b in tokens:
            y = lin.gemv(x[:b], m, y_dtype=aq.AQ_F32)
            assert np.all(np.abs(U.to_f64(y) - ref[:b]) <= bound[:b]), "m=%d batch=%d" % (m, b)
            assert np.array_equal(U.to_f64(lin.gemv(x[:b], m, y_dtype=aq.AQ_F32)), U.to_f64(y))
