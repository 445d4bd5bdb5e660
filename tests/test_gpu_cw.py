"""The codeword tensor-core GEMV (gemv_cw: 2..16 tokens with 4-bit codes, 3..16 with 8-bit codes;
y = x W_m^T of Sec. 2.2 with the prefix reconstruction of Sec. 3.2 / Sec. 5) where it can go wrong:
ragged row blocks and slices, fewer units than warps, clusters that split a row block's units, one
and two token tiles, both copy counts of the staged books, mixed operand types, weights that are
not marked static.

Tolerance: the operands are exact (values within 2^29 of the largest), so the error is that of the
fp32 sums: a warp's accumulator takes at most 16 multiplies of 16 inputs per (slice, book) unit, each
rounding by at most 2^-23 of sum |x||C|, and 16 warps and up to 8 CTAs are added after that. With at
most 33 slices x 8 books over 16 warps that is below (17 * 16 + 24) * 2^-23 < 2^-14 of
A = |s| sum_i |x_i| sum_k |C_k|_i, doubled for the scaled operands' smallest values."""
import numpy as np
import pytest
import torch

import aq_testutil as U
import oracle
import paper_2606_12876_gb300 as aq
import workloads
from paper_2606_12876_gb300.linear import AQLinear, x_to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    U.require_gpu()


def _widen(bits, dt):
    b = np.asarray(bits, np.uint16)
    return (b.view(np.float16) if dt == "f16" else (b.astype(np.uint32) << 16).view(np.float32)).astype(np.float64)


@pytest.mark.parametrize("out,inp,M,B,bdt,xdt", [
    (33, 264, 2, 8, "f16", "f16"),      # two row blocks, a slice with one group, fewer units than warps
    (1024, 1024, 3, 8, "f16", "bf16"),  # clusters
    (5000, 520, 5, 8, "bf16", "f16"),   # several row blocks per CTA, four copies of the books
    (96, 8200, 8, 8, "bf16", "bf16"),   # 33 slices, eight books
    (200, 2056, 4, 4, "f16", "bf16"),   # 4-bit codes
    (1, 8, 1, 4, "bf16", "f16"),        # one output, one group
])
def test_cw_edges(out, inp, M, B, bdt, xdt):
    layer = workloads.make_layer(out, inp, G=8, M=M, B=B, book_dtype=bdt, book_std=0.05,
                                 scale_dtype=bdt, seed=out + M)
    x_bits = workloads.make_x(16, inp, xdt, seed=inp)
    lin = AQLinear.from_layer(layer)
    x = x_to_device(x_bits, xdt)
    absl = dict(layer, books=np.asarray(layer["books"], np.uint16) & 0x7fff,
                scales=np.asarray(layer["scales"], np.uint16) & 0x7fff)
    X = np.abs(_widen(x_bits, xdt))
    for m in sorted({1, M - 1, M} - {0}):
        ref = oracle.product_exact(layer, x_bits, xdt, m)
        bound = 2.0 ** -13 * (X @ np.abs(oracle.reconstruct_exact(absl, m)).T)
        for b in (2, 3, 8, 9, 16):
            y = U.to_f64(lin.gemv(x[:b], m, y_dtype=aq.AQ_F32))
            assert np.all(np.abs(y - ref[:b]) <= bound[:b]), "m=%d batch=%d" % (m, b)
            lin.layout.flags = 0        # the same bits when the weights are read after the grid wait
            z = lin.gemv(x[:b], m, y_dtype=aq.AQ_F32)
            lin.layout.flags = aq.AQ_LAYOUT_STATIC_WEIGHTS
            assert np.array_equal(U.to_f64(z), y), "m=%d batch=%d, weights not static" % (m, b)
        y_prev = torch.ones(4, out, dtype=torch.float32, device="cuda")
        inc = U.to_f64(lin.refine(x[:4], m, y_prev)) - 1.0
        prev = oracle.product_exact(layer, x_bits[:4], xdt, m - 1) if m > 1 else 0.0
        assert np.all(np.abs(inc - (ref[:4] - prev)) <= bound[:4] + 2.0 ** -22 * (1 + np.abs(ref[:4])))


def test_cw_token_magnitudes():
    """fp16 books with bf16 activations far outside fp16's range, and tokens of widely different
    magnitude: every token keeps fp32 precision relative to its own terms."""
    layer = workloads.make_layer(160, 1032, G=8, M=3, B=8, book_dtype="f16", book_std=0.05, seed=1)
    rng = np.random.Generator(np.random.PCG64(2))
    xv = rng.standard_normal((6, 1032)).astype(np.float32)
    xv *= np.array([1e30, 1e-30, 1.0, 1e6, 0.0, 1e-6], np.float32)[:, None]
    x_bits = workloads.to_bits(xv, "bf16")
    lin = AQLinear.from_layer(layer)
    absl = dict(layer, books=np.asarray(layer["books"], np.uint16) & 0x7fff)
    y = U.to_f64(lin.gemv(x_to_device(x_bits, "bf16"), 3, y_dtype=aq.AQ_F32))
    bound = 2.0 ** -13 * (np.abs(_widen(x_bits, "bf16")) @ np.abs(oracle.reconstruct_exact(absl, 3)).T)
    assert np.all(np.abs(y - oracle.product_exact(layer, x_bits, "bf16", 3)) <= bound)
