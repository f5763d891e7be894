"""Inverted-residual blocks as one kernel: the depthwise walk's columns, strips and lanes (hidden chunks of 64, 48, 32 and 16
channels), both strides, maps smaller than a tile, ragged tiles, many tiles per CTA, one SM, blocks without an expansion layer,
wide outputs (issued as two halves, direct stores)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_05630_b200 import binding as B
from tests import gpu_util as G
from tests.test_gpu_parity import _conv, _mk

# (n, h, w, cin, hidden (0: no expansion layer), cout, stride)
CASES = [
    (2, 14, 14, 24, 144, 24, 1),       # last chunk of 16 channels, residual
    (1, 15, 17, 16, 96, 24, 2),        # last chunk of 32 channels, odd sizes
    (3, 7, 7, 40, 240, 64, 1),         # last chunk of 48 channels
    (2, 9, 33, 32, 192, 32, 1),        # wide and flat, residual
    (1, 3, 2, 8, 16, 8, 1),            # smaller than any tile
    (5, 23, 21, 64, 64, 128, 2),
    (2, 13, 29, 32, 0, 16, 1),         # no expansion layer
    (1, 20, 20, 96, 0, 96, 1),         # no expansion layer, two chunks, residual
    (1, 7, 7, 160, 960, 320, 1),       # three input planes, C_out > 256
    (2, 10, 12, 72, 288, 384, 1),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "n%d_%dx%d_%d_%d_%d_s%d" % c)
def test_block(case):
    n, h, w, cin, hid, cout, stride = case
    layers = [_conv(cin, hid, 1, act="relu6")] if hid else []
    mid = hid or cin
    layers.append(_conv(mid, mid, 3, stride=stride, act="relu6", groups=mid, op="dwconv", src=len(layers) - 1))
    layers.append(_conv(mid, cout, 1, act="none", src=len(layers) - 1, res_src=-1 if stride == 1 and cin == cout else -2))
    sess, xd, ref = _mk(layers, "mb", n, h, w, cin)
    last = len(layers) - 1
    for s in (B.device_sm_count(), 7, 1):
        G.check_plan(sess, xd, ref, [last], [s], "block S=%d" % s)
        assert sess.kernels() == ["mbconv_tc"]
    sess.close()
