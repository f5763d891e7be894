"""3x3 layers whose ring stages carry a kernel column (conv_tc): tile widths of 8 to 64, ragged edges, pairs and pooling."""
import numpy as np
import pytest
import torch

from paper_2011_05630_b200 import networks as nw
from paper_2011_05630_b200.runtime import Session

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,cout,n,h,w,act,pool,res", [
    (64, 64, 32, 56, 56, "relu", 0, False),      # the shape of a residual network's first 3x3 layers
    (64, 64, 5, 97, 131, "relu6", 0, True),      # wider than a tile, odd sizes, residual
    (64, 64, 3, 150, 202, "relu", 2, False),     # pooled, no multiple of the tile
    (128, 128, 7, 61, 59, "none", 2, True),      # pooled with a residual, odd map
    (128, 192, 9, 33, 47, "relu", 0, False),     # channel tiles of 64
    (64, 24, 11, 75, 90, "relu", 0, False),      # narrow output, padded to 32
    (192, 256, 24, 14, 14, "relu", 0, False),    # small maps
    (256, 256, 8, 28, 28, "relu", 2, False),
])
def test_kernel_columns(cin, cout, n, h, w, act, pool, res):
    layers = [nw._layer("conv", cin, cin, 1)] if res else []
    layers.append(nw._layer("conv", cin, cout, 3, act=act, pool=pool, res_src=0 if res else -2, src=-1 if res else None))
    layers = nw._finish(layers)
    g = torch.Generator().manual_seed(cin + cout + h)
    params = []
    for l in layers:
        k = l["kh"]
        params.append(((torch.randn(l["cout"], k, k, l["cin"], generator=g) * (k * k * l["cin"]) ** -0.5).half().numpy(),
                       (torch.randn(l["cout"], generator=g) * 0.1).numpy().astype(np.float32)))
    x = (torch.rand(n, h, w, cin, generator=g) * 2 - 1).half()
    s = Session(layers, params, n, h, w, cin)
    s.set_plan()
    y = s.run(x.cuda()).float().cpu()
    t = x.float().cuda().permute(0, 3, 1, 2)
    conv = lambda t, i: torch.nn.functional.conv2d(t, torch.from_numpy(params[i][0]).float().cuda().permute(0, 3, 1, 2),
                                                   torch.from_numpy(params[i][1]).cuda(), padding=layers[i]["pad"])
    torch.backends.cudnn.allow_tf32 = False
    r = conv(t, 0).half().float() if res else None
    ref = conv(t, len(layers) - 1)
    ref = ref + r if res else ref
    ref = ref if act == "none" else (ref.clamp(min=0) if act == "relu" else ref.clamp(0, 6))
    if pool:
        ref = torch.nn.functional.max_pool2d(ref, 2)
    ref = ref.permute(0, 2, 3, 1).cpu()
    s.close()
    assert y.shape == ref.shape
    # one rounding to fp16 (2^-11 of a value), at most another one of the residual, and fp32 sums of up to 2304 products of
    # values below one in another order (far below 2^-11)
    err = (y - ref).abs()
    assert bool((err <= 2 ** -10 * ref.abs() + 2 ** -10).all()), float(err.max())
