"""aq_gemv_group at 2..16 tokens, where layers share launches of the one-kernel forms (gemv_cw, gemm_ts): each
output equals the layer's own aq_gemv call bit for bit, over layers of very different heights (own
clusters, one row, none), both code widths, mixed and equal splits of K, and both operand mixes."""
import numpy as np
import pytest
import torch

import aq_testutil as U
import paper_2606_12876_gb300 as aq
import workloads
from paper_2606_12876_gb300.linear import AQLinear, gemv_group, x_to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def gpu():
    U.require_gpu()


@pytest.mark.parametrize("outs,inp,M,B,bdt,xdt", [
    ((4096, 1024, 1024), 4096, 3, 8, "f16", "bf16"),
    ((4100, 4100), 1032, 4, 8, "bf16", "bf16"),
    ((1, 33, 640, 5000), 520, 2, 8, "f16", "f16"),
    ((2048, 96), 2056, 4, 4, "f16", "bf16"),
    ((12288, 64, 300), 2048, 5, 8, "bf16", "f16"),
])
def test_group_equals_single_calls(outs, inp, M, B, bdt, xdt):
    lins = [AQLinear.from_layer(workloads.make_layer(o, inp, G=8, M=M, B=B, book_dtype=bdt, scale_dtype=bdt, seed=o + i))
            for i, o in enumerate(outs)]
    x = x_to_device(workloads.make_x(16, inp, xdt, seed=inp), xdt)
    for m in sorted({1, M}):
        for b in (2, 3, 8, 9, 16):
            ys = gemv_group(lins, x[:b], m, y_dtype=aq.AQ_F32)
            for lin, y in zip(lins, ys):
                assert torch.equal(y, lin.gemv(x[:b], m, y_dtype=aq.AQ_F32)), "out=%d m=%d batch=%d" % (lin.out, m, b)
            lins[-1].layout.flags = 0          # one layer's weights not marked static
            zs = gemv_group(lins, x[:b], m, y_dtype=aq.AQ_F32)
            lins[-1].layout.flags = aq.AQ_LAYOUT_STATIC_WEIGHTS
            assert all(torch.equal(y, z) for y, z in zip(ys, zs)), "m=%d batch=%d, not static" % (m, b)
