"""The fp32 error of the products whose weights are exact and whose sums are fp32 (gemv_cw at up to four tokens,
with one book over several units of a warp, and with 4-bit codes; y = x W_m^T of Sec. 2.2 with the prefix reconstruction of Sec. 3.2 / Sec. 5),
measured against the table form in fp32: per group and book a chain of eight fused multiply-adds, 32 groups
added in order, then the slices' and books' sums in order.

Tolerance: 1.2 times the table form's relative error. The table form rounds 8 + 32 times per slice and book,
in order, and then once per slice and book; gemv_cw adds 16 multiplies' sums in pairs, then eight of
those in order, then pairs of warps: less than half of that variance. A multiply truncates its sum of 16
products, which is at most one unit in the last place of it and shrinks y by 0.5 to 1 x 2^-24 of its value
on average; the table form's error is about 1.5 x 2^-24, so both together stay below 1.2 times it. (Chains of
eight multiplies without additions in between measured 2 times the table form, longer ones 3 to 40 times.)

With one book from five tokens, one unit of a warp is one chain of 16 truncating multiplies: each truncation is on
average half to one unit in the last place (2^-24 to 2^-23) of a partial sum that grows with the square root of
its terms, on average two thirds of the unit's: 16 * 0.75 * 2^-24 * 2/3 = 4.8e-7 of y."""
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


def table_form(layer, X, ks):
    """sum_k of books ks, fp32 as above, times the row scales. X: [tokens][in] float64 of 16-bit values."""
    out, ng = layer["out"], layer["in"] // 8
    books = _widen(layer["books"], layer["book_dtype"])
    xg = X.reshape(len(X), ng, 8)
    total = np.zeros((len(X), out), np.float32)
    for s0 in range(0, ng, 32):
        for k in ks:
            codes = layer["codes"][:, s0:s0 + 32, k]                       # [out][groups]
            part = np.zeros((len(X), out), np.float32)
            for g in range(codes.shape[1]):
                T = np.zeros((len(X), books.shape[1]), np.float32)          # one table entry per codeword
                for e in range(8):
                    T = (T.astype(np.float64) + xg[:, s0 + g, e, None] * books[k][None, :, e]).astype(np.float32)
                part += T[:, codes[:, g]]
            total += part
    return total * _widen(layer["scales"], layer["scale_dtype"]).astype(np.float32)


def rel(y, ref):
    return np.linalg.norm(y - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("bdt,xdt", [("f16", "f16"), ("f16", "bf16"), ("bf16", "bf16"), ("bf16", "f16")])
@pytest.mark.parametrize("out,inp,M,B,batches,one_book", [
    (1024, 1024, 2, 8, (1, 3, 4), ()),                  # one kernel at one token as well; clusters
    (700, 4104, 3, 8, (4,), ()),                        # several units per warp, a ragged last slice
    (700, 4104, 3, 4, (2, 4, 16), (16,)),               # 4-bit codes
    (9000, 2048, 2, 8, (3,), ()),                       # several passes
    (5000, 4360, 2, 8, (), (5, 8, 9, 16)),              # one book, two units of some warps
])
def test_fp32_error(out, inp, M, B, batches, one_book, bdt, xdt):
    layer = workloads.make_layer(out, inp, G=8, M=M, B=B, book_dtype=bdt, book_std=0.02, scale_dtype=bdt, seed=out + M)
    x_bits = workloads.make_x(16, inp, xdt, seed=inp)
    X = _widen(x_bits, xdt)
    lin = AQLinear.from_layer(layer)
    x = x_to_device(x_bits, xdt)
    ref = oracle.product_exact(layer, x_bits, xdt, M)
    base = rel(table_form(layer, X[:4], range(M)), ref[:4]) if batches else 0.0
    for b in batches:
        err = rel(U.to_f64(lin.gemv(x[:b], M, y_dtype=aq.AQ_F32)), ref[:b])
        assert err <= 1.2 * base, "m=%d batch=%d: %.3g against %.3g" % (M, b, err, base)
    ref1 = oracle.product_exact(layer, x_bits, xdt, 1)
    base = rel(table_form(layer, X[:4], range(1)), ref1[:4])
    for b in one_book + batches:
        err = rel(U.to_f64(lin.gemv(x[:b], 1, y_dtype=aq.AQ_F32)), ref1[:b])
        assert err <= 1.2 * base, "m=1 batch=%d: %.3g against %.3g" % (b, err, base)
    ref2 = ref - oracle.product_exact(layer, x_bits, xdt, M - 1)     # the increment of the last book
    base = rel(table_form(layer, X[:4], [M - 1]), ref2[:4])
    for b in one_book:
        err = rel(U.to_f64(lin.refine(x[:b], M, None)), ref2[:b])
        assert err <= 1.2 * base, "refine batch=%d: %.3g against %.3g" % (b, err, base)


@pytest.mark.parametrize("bdt,xdt", [("f16", "f16"), ("f16", "bf16"), ("bf16", "bf16"), ("bf16", "f16")])
@pytest.mark.parametrize("out,inp", [(1024, 1024), (259, 2568), (5000, 4096)])
def test_one_book_one_unit(out, inp, bdt, xdt):
    layer = workloads.make_layer(out, inp, G=8, M=2, B=8, book_dtype=bdt, book_std=0.02, scale_dtype=bdt, seed=out)
    x_bits = workloads.make_x(16, inp, xdt, seed=inp)
    lin = AQLinear.from_layer(layer)
    x = x_to_device(x_bits, xdt)
    ref = oracle.product_exact(layer, x_bits, xdt, 1)
    for b in (5, 8, 9, 16):
        assert rel(U.to_f64(lin.gemv(x[:b], 1, y_dtype=aq.AQ_F32)), ref[:b]) <= 4.8e-7, "batch=%d" % b
