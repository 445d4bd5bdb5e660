"""Three and four tokens on layers of more row blocks than SMs, where the table kernel with two 64 KiB tables takes
the call from gemv_cw (y = x W_m^T of Sec. 2.2 with the prefix reconstruction of Sec. 3.2 / Sec. 5): the
kernel that runs, ragged rows and slices, both operand mixes, refinement, groups equal to single calls.

Tolerance: exact operands and fp32 sums, as derived in test_gpu_fp32_sums (1.2 times the table form's relative
error there; this is the table form) and, per element, 2^-13 of A = |s| sum_i |x_i| sum_k |C_k|_i."""
import numpy as np
import pytest
import torch

import aq_testutil as U
import oracle
import paper_2606_12876_gb300 as aq
import workloads
from graph_kernels import kernels
from paper_2606_12876_gb300.linear import AQLinear, gemv_group, x_to_device
from test_gpu_cw import _widen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    U.require_gpu()


def names(call):
    return [k[0] for k in kernels(call)]


@pytest.mark.parametrize("bdt,xdt", [("f16", "bf16"), ("bf16", "f16"), ("f16", "f16"), ("bf16", "bf16")])
def test_tables_for_four_tokens(bdt, xdt):
    out, inp, M = 4900, 3080, 5
    layer = workloads.make_layer(out, inp, G=8, M=M, B=8, book_dtype=bdt, book_std=0.05, scale_dtype=bdt, seed=1)
    x_bits = workloads.make_x(4, inp, xdt, seed=2)
    lin = AQLinear.from_layer(layer)
    x = x_to_device(x_bits, xdt)
    absl = dict(layer, books=np.asarray(layer["books"], np.uint16) & 0x7fff,
                scales=np.asarray(layer["scales"], np.uint16) & 0x7fff)
    ref = oracle.product_exact(layer, x_bits, xdt, 4)
    A = np.abs(_widen(x_bits, xdt)) @ np.abs(oracle.reconstruct_exact(absl, 4)).T
    y = torch.empty(4, out, device="cuda")
    for b in (3, 4):
        if torch.cuda.get_device_properties(0).multi_processor_count == 152:
            assert names(lambda: lin.gemv(x[:b], 4, y=y[:b], y_dtype=aq.AQ_F32)) == ["gemv_lut_kernel", "splitk_reduce_kernel"]
            assert names(lambda: lin.gemv(x[:b], 5, y=y[:b], y_dtype=aq.AQ_F32)) == ["gemv_cw_kernel"]
        got = U.to_f64(lin.gemv(x[:b], 4, y_dtype=aq.AQ_F32))
        assert np.all(np.abs(got - ref[:b]) <= 2.0 ** -13 * A[:b])
        assert np.linalg.norm(got - ref[:b]) <= 2e-7 * np.linalg.norm(ref[:b])
        other = AQLinear.from_layer(workloads.make_layer(96, inp, G=8, M=M, B=8, book_dtype=bdt, scale_dtype=bdt, seed=3))
        ys = gemv_group([lin, other], x[:b], 4, y_dtype=aq.AQ_F32)
        assert np.array_equal(U.to_f64(ys[0]), got)
        assert torch.equal(ys[1], other.gemv(x[:b], 4, y_dtype=aq.AQ_F32))


def test_refinement():
    """One book's increment over 49 slices."""
    layer = workloads.make_layer(4900, 12296, G=8, M=2, B=8, book_dtype="f16", book_std=0.05, scale_dtype="f16", seed=4)
    x_bits = workloads.make_x(4, 12296, "f16", seed=5)
    lin = AQLinear.from_layer(layer)
    x = x_to_device(x_bits, "f16")
    ref = oracle.product_exact(layer, x_bits, "f16", 2) - oracle.product_exact(layer, x_bits, "f16", 1)
    got = U.to_f64(lin.refine(x, 2, None))
    assert np.linalg.norm(got - ref) <= 2e-7 * np.linalg.norm(ref)
    y = lin.gemv(x, 1, y_dtype=aq.AQ_F32)
    full = U.to_f64(lin.refine(x, 2, y, y=y))
    ref2 = oracle.product_exact(layer, x_bits, "f16", 2)
    assert np.linalg.norm(full - ref2) <= 3e-7 * np.linalg.norm(ref2)
