"""aq_gemv_group with layers of different forms at one token (8-bit codes: the table kernel for tall layers, gemv_cw for
small ones): the layers of a form share launches, and each output equals the layer's own call bit for bit
(y = x W_m^T of Sec. 2.2)."""
import pytest
import torch

import aq_testutil as U
import paper_2606_12876_gb300 as aq
import workloads
from graph_kernels import kernels
from paper_2606_12876_gb300.linear import AQLinear, gemv_group, x_to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    U.require_gpu()


TABLES, CW = ["gemv_lut_kernel", "splitk_reduce_kernel"], ["gemv_cw_kernel"]


@pytest.mark.parametrize("outs,inp,m,launches", [
    ((4096, 1024, 1024), 1024, 2, CW + TABLES),           # one tall layer, two small ones
    ((1024, 4096, 2080, 64), 1024, 2, CW + TABLES),       # two and two, in turn
    ((1024, 1024, 512), 1024, 2, CW),
    ((4096, 4096, 0, 8192), 1032, 1, TABLES),             # an empty layer among tall ones
])
@pytest.mark.parametrize("xdt", ["f16", "bf16"])
def test_mixed_group(outs, inp, m, launches, xdt):
    lins = [AQLinear.from_layer(workloads.make_layer(max(o, 1), inp, G=8, M=2, B=8, book_dtype="f16", scale_dtype="f16",
                                                     seed=i)) for i, o in enumerate(outs)]
    for lin, o in zip(lins, outs):
        if o == 0:
            lin.layout.out_features = lin.out = 0
    x = x_to_device(workloads.make_x(1, inp, xdt, seed=9), xdt)
    ys = [torch.full((1, o), 7.0, device="cuda") for o in outs]
    assert [k[0] for k in kernels(lambda: gemv_group(lins, x, m, ys=ys, y_dtype=aq.AQ_F32))] == launches
    for lin, o, y in zip(lins, outs, gemv_group(lins, x, m, y_dtype=aq.AQ_F32)):
        if o:
            assert torch.equal(y, lin.gemv(x, m, y_dtype=aq.AQ_F32)), "out=%d" % o
