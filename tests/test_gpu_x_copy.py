"""aq_gemm's fp16 copy of bf16 activations at the row lengths where its launch changes: rows of one 16-byte
piece, held in registers by 256, 512 and 1024 threads, and longer than the registers hold; rows of zeros and of
very different magnitudes; more rows than CTAs (y = x W_m^T of Sec. 2.2).

Tolerance: a weight is rounded once to fp16 (2^-11 of sum_k |C_k|), the rest are fp32 sums of at most 2^16
terms in chains of at most 2^9 (below 2^-13 of A = |s| sum_i |x_i| sum_k |C_k|_i); the scaled activations are
exact within 2^29 of the row's largest."""
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


@pytest.mark.parametrize("inp,tokens", [(8, 17), (8192, 18), (8200, 19), (16392, 17), (32776, 21), (40960, 17), (264, 1300)])
def test_row_lengths(inp, tokens):
    out, M = 40, 2
    layer = workloads.make_layer(out, inp, G=8, M=M, B=8, book_dtype="f16", book_std=0.05, scale_dtype="f16", seed=inp)
    rng = np.random.Generator(np.random.PCG64(inp))
    v = rng.standard_normal((tokens, inp)).astype(np.float32) * 10.0 ** rng.uniform(-4, 4, (tokens, 1)).astype(np.float32)
    v[3] = 0.0
    x_bits = workloads.to_bits(v, "bf16")
    lin = AQLinear.from_layer(layer)
    x = x_to_device(x_bits, "bf16")
    absl = dict(layer, books=np.asarray(layer["books"], np.uint16) & 0x7fff,
                scales=np.asarray(layer["scales"], np.uint16) & 0x7fff)
    ref = oracle.product_exact(layer, x_bits, "bf16", M)
    bound = (2.0 ** -11 + 2.0 ** -13) * (np.abs(_widen(x_bits, "bf16")) @ np.abs(oracle.reconstruct_exact(absl, M)).T)
    y = U.to_f64(lin.gemm(x, M, y_dtype=aq.AQ_F32))
    assert np.all(np.abs(y - ref) <= bound)
