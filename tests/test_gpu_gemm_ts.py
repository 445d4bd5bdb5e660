"""The tensor-memory GEMM (gemm_ts: 9..2047 tokens, up to four books; y = x W_m^T of Sec. 2.2 with the
prefix reconstruction of Sec. 3.2 / Sec. 5) at the edges of its tiles: rows that end inside a row
quarter, tiles of one to four quarters, clusters with ranks that have few slices or none, a last slice with
few groups, token counts around multiples of 16 and of the 256-token tile, output rows that allow no
16-byte stores, every output type, 4-bit codes, weights that are not marked static.

Every weight is rounded once to fp16 (2^-11 relative), the rest is fp32 accumulation, so
|y - y_exact| <= (2^-11 + 2^-13) |s| sum_i |x_i| sum_k |C_k|_i, plus one rounding of a 16-bit y; inputs
chosen as in test_gpu_exact give the oracle's fp64 product bit for bit. Which kernel a call runs is the
library's choice: the bound holds for all of them."""
import numpy as np
import pytest

import aq_testutil as U
import oracle
import paper_2606_12876_gb300 as aq
import workloads
from paper_2606_12876_gb300.linear import AQLinear, x_to_device
from test_gpu_exact import assert_exact, exact_layer, exact_x

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    U.require_gpu()


def _widen(bits, dt):
    b = np.asarray(bits, np.uint16)
    return (b.view(np.float16) if dt == "f16" else (b.astype(np.uint32) << 16).view(np.float32)).astype(np.float64)


@pytest.mark.parametrize("out,inp,M,B,bdt,xdt,tokens", [
    (33, 264, 2, 8, "f16", "bf16", (17, 33)),          # one row past a quarter, one group past a slice
    (1000, 2056, 4, 8, "bf16", "bf16", (17, 100, 256)),   # nine slices: uneven clusters
    (4100, 1024, 3, 8, "f16", "f16", (48, 257)),       # out % 8 != 0: no 16-byte stores; two token tiles
    (300, 520, 4, 4, "f16", "bf16", (31, 300)),        # 4-bit codes
    (2048, 4096, 1, 8, "bf16", "f16", (16, 240)),
])
def test_ts_edges(out, inp, M, B, bdt, xdt, tokens):
    layer = workloads.make_layer(out, inp, G=8, M=M, B=B, book_dtype=bdt, book_std=0.05,
                                 scale_dtype=bdt, seed=out + M)
    x_bits = workloads.make_x(max(tokens), inp, xdt, seed=inp)
    lin = AQLinear.from_layer(layer)
    x = x_to_device(x_bits, xdt)
    absl = dict(layer, books=np.asarray(layer["books"], np.uint16) & 0x7fff,
                scales=np.asarray(layer["scales"], np.uint16) & 0x7fff)
    for m in sorted({1, M}):
        ref = oracle.product_exact(layer, x_bits, xdt, m)
        bound = (2.0 ** -11 + 2.0 ** -13) * (np.abs(_widen(x_bits, xdt)) @ np.abs(oracle.reconstruct_exact(absl, m)).T)
        for t in tokens:
            for yd, ulp in ((aq.AQ_F32, 0.0), (aq.AQ_F16, 2.0 ** -11), (aq.AQ_BF16, 2.0 ** -8)):
                y = U.to_f64(lin.gemm(x[:t], m, y_dtype=yd) if t > 16 else lin.gemv(x[:t], m, y_dtype=yd))
                excess = np.abs(y - ref[:t]) - bound[:t] * (1 + ulp) - ulp * np.abs(ref[:t]) - 2.0 ** -24
                assert np.all(excess <= 0), "m=%d tokens=%d y type %d: %d beyond" % (m, t, yd, int(np.sum(excess > 0)))
            if t > 16:
                a = lin.gemm(x[:t], m, y_dtype=aq.AQ_F32)
                lin.layout.flags = 0        # the same bits when the weights are read after the grid wait
                b = lin.gemm(x[:t], m, y_dtype=aq.AQ_F32)
                lin.layout.flags = aq.AQ_LAYOUT_STATIC_WEIGHTS
                assert np.array_equal(U.to_f64(a), U.to_f64(b)), "m=%d tokens=%d, weights not static" % (m, t)


@pytest.mark.parametrize("out,inp,tokens", [(96, 16384, 40), (3000, 1032, 130), (512, 2048, 1100)])
def test_ts_exact(out, inp, tokens):
    layer = exact_layer(out, inp, 4, 8, "f16", seed=out)
    lin = AQLinear.from_layer(layer)
    x_bits = exact_x(tokens, inp, "bf16", seed=inp)
    x = x_to_device(x_bits, "bf16")
    for m in (2, 4):
        assert_exact(lin.gemm(x, m, y_dtype=aq.AQ_F32), oracle.product_exact(layer, x_bits, "bf16", m), "m=%d" % m)
