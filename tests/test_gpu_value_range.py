"""The power-of-two scalings of the mixed-type kernels (gemv_cw, gemm_ts, the prefill GEMM) at the ends of
bf16's range, where y is an ordinary value: activations and codebooks of about 2^120 and of bf16's
smallest normal values, and products of very large and very small ones; y = x W_m^T of Sec. 2.2 with the
prefix reconstruction of Sec. 3.2 / Sec. 5.

Tolerance: a weight may be rounded once to fp16 (2^-11 of sum_k |C_k|), the rest are fp32 sums (below
2^-13 of A = |s| sum_i |x_i| sum_k |C_k|_i, as derived in test_gpu_cw); results below fp32's normal range
are rounded to multiples of 2^-149 by each of fewer than 2^9 additions of partial sums."""
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


def scaled_layer(out, inp, M, B, bdt, e, seed):
    """A layer with codebooks of standard deviation 0.05 * 2^e."""
    layer = workloads.make_layer(out, inp, G=8, M=M, B=B, book_dtype=bdt, book_std=0.05, scale_dtype=bdt, seed=seed)
    if e:
        layer["books"] = workloads.to_bits((_widen(layer["books"], bdt) * 2.0 ** e).astype(np.float32), bdt)
    return layer


def scaled_x(tokens, inp, xdt, e, seed):
    v = np.random.Generator(np.random.PCG64(seed)).standard_normal((tokens, inp)) * 2.0 ** e
    return workloads.to_bits(v.astype(np.float32), xdt)


def check(layer, x_bits, xdt, m, batches, rows=slice(None)):
    """Every product entry point at the token counts `batches`, rows `rows` of the outputs."""
    lin = AQLinear.from_layer(layer)
    x = x_to_device(x_bits, xdt)
    absl = dict(layer, books=np.asarray(layer["books"], np.uint16) & 0x7fff,
                scales=np.asarray(layer["scales"], np.uint16) & 0x7fff)
    ref = oracle.product_exact(layer, x_bits, xdt, m)[:, rows]
    A = np.abs(_widen(x_bits, xdt)) @ np.abs(oracle.reconstruct_exact(absl, m))[rows].T
    assert np.abs(ref).max() < 2.0 ** 127
    for b in batches:
        call = lin.gemv if b <= 16 else lin.gemm
        y = U.to_f64(call(x[:b], m, y_dtype=aq.AQ_F32))[:, rows]
        bad = ~(np.abs(y - ref[:b]) <= (2.0 ** -11 + 2.0 ** -13) * A[:b] + 2.0 ** -140)
        assert not bad.any(), "m=%d tokens=%d: %d of %d outputs, e.g. %r for %r" % (
            m, b, int(bad.sum()), bad.size, y[bad][0], ref[:b][bad][0])


TOKENS = (1, 2, 3, 8, 9, 16, 17, 100)


@pytest.mark.parametrize("e", [120, 113, -112, -122])
@pytest.mark.parametrize("out,inp,M,B", [(40, 264, 3, 8), (700, 2056, 5, 8), (72, 520, 4, 4)])
def test_activation_range(out, inp, M, B, e):
    layer = scaled_layer(out, inp, M, B, "f16", 0, seed=out)
    x_bits = scaled_x(100, inp, "bf16", e, seed=inp)
    for m in sorted({1, M}):
        check(layer, x_bits, "bf16", m, TOKENS)


@pytest.mark.parametrize("e", [119, -118])
@pytest.mark.parametrize("out,inp,M,B", [(40, 264, 3, 8), (700, 2056, 5, 8), (72, 520, 4, 4)])
def test_codebook_range(out, inp, M, B, e):
    layer = scaled_layer(out, inp, M, B, "bf16", e, seed=out)
    x_bits = scaled_x(100, inp, "f16", 0, seed=inp)
    for m in sorted({1, M}):
        check(layer, x_bits, "f16", m, TOKENS)


@pytest.mark.parametrize("ew,ex", [(0, 112), (-118, 118), (100, -112), (-60, 100)])
@pytest.mark.parametrize("out,inp,M,B", [(40, 264, 3, 8), (700, 2056, 5, 8), (72, 520, 4, 4)])
def test_large_times_small(out, inp, M, B, ew, ex):
    """bf16 books and activations whose scale factors together exceed the range of either."""
    layer = scaled_layer(out, inp, M, B, "bf16", ew, seed=out)
    x_bits = scaled_x(100, inp, "bf16", ex, seed=inp)
    for m in sorted({1, M}):
        check(layer, x_bits, "bf16", m, TOKENS)


def test_large_times_small_dense():
    """The same where W_m is decoded first (2048 tokens and more)."""
    layer = scaled_layer(72, 264, 3, 8, "bf16", -118, seed=1)
    check(layer, scaled_x(2048, 264, "bf16", 118, seed=2), "bf16", 3, (2048,))


@pytest.mark.parametrize("bdt,xdt", [("f16", "f16"), ("f16", "bf16"), ("bf16", "f16"), ("bf16", "bf16")])
@pytest.mark.parametrize("out,inp,M,B", [(40, 256, 3, 8), (700, 2048, 5, 8), (72, 512, 4, 4)])
def test_infinite_codeword(out, inp, M, B, bdt, xdt):
    """An infinite entry in a book: rows that use its codeword are not finite, the others keep their values
    (codeword 0 stays finite: the positions past a row's last group hold code 0)."""
    layer = scaled_layer(out, inp, M, B, bdt, 0, seed=out)
    used = np.zeros(out, bool)
    used[::9] = True
    layer["codes"] = np.where(layer["codes"] == 7, 6, layer["codes"]).astype(layer["codes"].dtype)
    layer["codes"][used, 3, 0] = 7
    layer["books"] = np.array(layer["books"], np.uint16)
    layer["books"][0, 7, 2] = 0x7c00 if bdt == "f16" else 0x7f80
    x_bits = scaled_x(100, inp, xdt, 0, seed=inp)
    finite = dict(layer, books=layer["books"].copy())
    finite["books"][0, 7, 2] = 0
    lin = AQLinear.from_layer(layer)
    x = x_to_device(x_bits, xdt)
    absl = dict(finite, books=finite["books"] & 0x7fff, scales=np.asarray(layer["scales"], np.uint16) & 0x7fff)
    for m in sorted({1, M}):
        ref = oracle.product_exact(finite, x_bits, xdt, m)
        A = np.abs(_widen(x_bits, xdt)) @ np.abs(oracle.reconstruct_exact(absl, m)).T
        for b in TOKENS:
            y = U.to_f64((lin.gemv if b <= 16 else lin.gemm)(x[:b], m, y_dtype=aq.AQ_F32))
            bad = ~(np.abs(y - ref[:b]) <= (2.0 ** -11 + 2.0 ** -13) * A[:b])
            assert not bad[:, ~used].any(), "m=%d tokens=%d: %d outputs of rows that do not use it" % (
                m, b, int(bad[:, ~used].sum()))
            assert not np.isfinite(y[:, used]).any(), "m=%d tokens=%d" % (m, b)
