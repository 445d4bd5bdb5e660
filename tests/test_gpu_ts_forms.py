"""Every form of the tensor-memory GEMM (gemm_ts: tiles of one to four row quarters, clusters of one to eight CTAs
that split K, eight or four copies of a book): the form that a call takes, read from a captured graph, and its
result on exact arithmetic (see test_gpu_exact), bit for bit (y = x W_m^T of Sec. 2.2 with the prefix
reconstruction of Sec. 3.2 / Sec. 5). Also which kernel the GEMV takes at the edges of its rules. The forms are
those of 152 SMs; on another number only the results are compared."""
import pytest
import torch

import aq_testutil as U
import oracle
import paper_2606_12876_gb300 as aq
import workloads
from graph_kernels import kernels
from paper_2606_12876_gb300.linear import AQLinear, x_to_device
from test_gpu_exact import assert_exact, exact_layer, exact_x

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    U.require_gpu()


def all_sms():
    return torch.cuda.get_device_properties(0).multi_processor_count == 152


@pytest.mark.parametrize("quarters,cluster,out,inp,m,tokens", [
    (1, 1, 33, 264, 2, 17), (1, 2, 33, 1032, 3, 17), (1, 4, 33, 2056, 4, 17), (1, 8, 33, 4104, 1, 17),
    (2, 1, 5000, 264, 3, 17), (2, 2, 3000, 1032, 4, 17), (2, 4, 2048, 2056, 1, 17), (2, 8, 300, 4104, 2, 17),
    (3, 1, 12000, 264, 4, 17), (3, 2, 5000, 1032, 1, 17), (3, 4, 3000, 2056, 2, 17), (3, 8, 700, 4104, 3, 17),
    (4, 1, 9000, 264, 1, 300), (4, 2, 9000, 1032, 2, 17), (4, 4, 4100, 2056, 3, 17), (4, 8, 1000, 4104, 4, 17),
    (3, 2, 5000, 4104, 5, 16), (3, 2, 5000, 1032, 6, 9), (2, 2, 4100, 8200, 7, 16), (3, 2, 5000, 1032, 8, 16),
])
def test_form(quarters, cluster, out, inp, m, tokens):
    layer = exact_layer(out, inp, max(m, 2), 8, "f16", seed=out)
    lin = AQLinear.from_layer(layer)
    x_bits = exact_x(tokens, inp, "bf16", seed=inp)
    x = x_to_device(x_bits, "bf16")
    y = torch.empty(tokens, out, device="cuda")
    call = lambda: (lin.gemm if tokens > 16 else lin.gemv)(x, m, y=y, y_dtype=aq.AQ_F32)
    if all_sms():
        copy, product = kernels(call)
        assert copy[0] == "bf16_rows_to_f16_kernel" and product[0] == "gemm_ts_kernel"
        assert product[1][:3] == (8, 0, m) and product[4] == cluster
        assert product[2][0] == cluster * -(-out // (32 * quarters)) and product[2][1] == -(-tokens // 256)
        assert product[3][0] == (576 if quarters == 4 else 512)
    y.fill_(0)
    call()
    assert_exact(y, oracle.product_exact(layer, x_bits, "bf16", m), "m=%d" % m)


@pytest.mark.parametrize("out,inp,m,B,batch,names", [
    (1024, 1024, 2, 8, 1, ["gemv_cw_kernel"]),                            # small: one kernel
    (2080, 1024, 2, 8, 1, ["gemv_lut_kernel", "splitk_reduce_kernel"]),   # more than 64 row blocks
    (1024, 1032, 2, 8, 1, ["gemv_lut_kernel", "splitk_reduce_kernel"]),   # more than eight units
    (1024, 1024, 2, 8, 2, ["gemv_lut_kernel", "splitk_reduce_kernel"]),
    (1024, 1024, 2, 8, 3, ["gemv_cw_kernel"]),
    (4096, 4096, 4, 8, 8, ["gemv_cw_kernel"]),
    (4096, 4096, 4, 8, 9, ["gemm_ts_kernel"]),
    (4096, 4096, 1, 8, 9, ["gemv_cw_kernel"]),                            # one book, fp32 y: exact weights, fp32 sums
    (14336, 2048, 1, 8, 16, ["gemm_ts_kernel"]),                          # one book, 16-bit y
    (1024, 1024, 4, 8, 16, ["gemv_cw_kernel"]),
    (1024, 1024, 4, 4, 1, ["gemv_lut4_kernel"]),
    (4096, 4096, 4, 4, 16, ["gemv_cw_kernel"]),                           # 4-bit codes: no rounded weights
])
def test_gemv_kernel(out, inp, m, B, batch, names):
    lin = AQLinear.from_layer(workloads.make_layer(out, inp, G=8, M=4, B=B, book_dtype="f16", scale_dtype="f16", seed=1))
    x = x_to_device(workloads.make_x(batch, inp, "f16", seed=2), "f16")
    yd = aq.AQ_F32 if m == 1 and names == ["gemv_cw_kernel"] else aq.AQ_F16
    y = torch.empty(batch, out, dtype=torch.float32 if yd == aq.AQ_F32 else torch.float16, device="cuda")
    if all_sms():
        assert [k[0] for k in kernels(lambda: lin.gemv(x, m, y=y, y_dtype=yd))] == names
    lin.gemv(x, m, y=y, y_dtype=yd)
    W = lin.decode(m).double()                # one rounding of a weight to fp16, one of y, fp32 sums
    ref, bound = x.double() @ W.t(), 2.0 ** -9 * (x.double().abs() @ W.abs().t())
    assert bool(((y.double() - ref).abs() <= bound + 1e-6).all())
