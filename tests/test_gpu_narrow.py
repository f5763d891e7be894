"""Pointwise layers with at most 64 input channels (conv_narrow): every width of its blocks, tails of pixels, residuals, and
both sides of the line to the tcgen05 kernels."""
import numpy as np
import pytest
import torch

from paper_2011_05630_b200 import networks as nw
from paper_2011_05630_b200.runtime import Session

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,n,h,w,act,res", [
    (8, 8, 1, 1, 1, "none", False), (16, 24, 3, 17, 13, "relu", False), (24, 24, 5, 31, 29, "relu6", True),
    (32, 16, 9, 112, 112, "none", False), (40, 32, 2, 33, 7, "relu", False), (64, 8, 1, 50, 51, "relu6", False),
    (64, 64, 7, 28, 28, "relu", True), (16, 96, 4, 56, 57, "relu6", False), (56, 192, 1, 15, 16, "none", False),
    (32, 256, 3, 20, 20, "relu", False), (64, 256, 3, 56, 56, "relu", False), (64, 256, 4, 56, 56, "relu", False), (64, 64, 33, 56, 56, "none", True)])
def test_pointwise(cin, cout, n, h, w, act, res):
    if res:
        layers = nw._finish([nw._layer("conv", cin, cout, 1, act=act, res_src=-1)])
    else:
        layers = nw._finish([nw._layer("conv", cin, cout, 1, act=act)])
    g = torch.Generator().manual_seed(cin * cout + n)
    wt = (torch.randn(cout, 1, 1, cin, generator=g) * cin ** -0.5).half()
    b = torch.randn(cout, generator=g) * 0.1
    x = (torch.rand(n, h, w, cin, generator=g) * 2 - 1).half()
    s = Session(layers, [(wt.numpy(), b.numpy())], n, h, w, cin)
    s.set_plan()
    y = s.run(x.cuda()).double().cpu()
    ref = x.double().reshape(-1, cin) @ wt.double().reshape(cout, cin).T + b.double()
    ref = ref.reshape(n, h, w, cout) + (x.double() if res else 0.0)
    ref = ref if act == "none" else (ref.clamp(min=0) if act == "relu" else ref.clamp(0, 6))
    s.close()
    # one rounding to fp16 (2^-11 of a value) and fp32 sums of 64 products below one (64 * 2^-24)
    err = (y - ref).abs()
    assert bool((err <= 2 ** -11 * ref.abs() + 2 ** -16).all()), float((err - 2 ** -11 * ref.abs()).max())
