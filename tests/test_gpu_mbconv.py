"""Inverted-residual blocks as one kernel: the depthwise walk's columns, strips and lanes (hidden chunks of 64, 48, 32 and 16
channels), both strides, maps smaller than a tile, ragged tiles, many tiles per CTA, one SM, blocks without an expansion layer,
wide outputs (issued as two halves, direct stores).  `test_block` takes the kernel that the sizes send a block to ("mbconv_tc" is the
group's kind: the persistent kernel, or on few images the one by clusters), `test_persistent_kernel` asks for the former by name."""
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


# (n, h, w, cin, hidden, cout, stride, activation): sizes at which the persistent kernel is the faster one on all SMs
PERSISTENT = [
    (33, 21, 19, 24, 144, 24, 1, "relu6"),      # last chunk of 16 channels, residual
    (60, 21, 19, 16, 80, 40, 2, "relu"),        # the same, stride 2
    (60, 21, 19, 32, 160, 32, 2, "relu6"),      # last chunk of 32
    (60, 21, 19, 40, 240, 40, 1, "relu6"),      # last chunk of 48, residual
    (17, 21, 19, 24, 48, 16, 2, "none"),        # that one alone
    (33, 21, 19, 64, 192, 64, 1, "none"),       # whole chunks, residual
    (17, 21, 19, 72, 208, 136, 1, "relu"),      # two input planes
    (9, 21, 19, 160, 320, 160, 1, "relu6"),     # three, residual
    (9, 21, 19, 200, 400, 24, 2, "none"),       # four
    (5, 21, 19, 136, 272, 320, 1, "relu6"),     # projection issued as two halves
    (9, 21, 19, 136, 272, 320, 2, "relu6"),
]


@pytest.mark.parametrize("case", PERSISTENT, ids=lambda c: "n%d_%dx%d_%d_%d_%d_s%d" % c[:7])
def test_persistent_kernel(case):
    n, h, w, cin, hid, cout, stride, act = case
    layers = [_conv(cin, hid, 1, act=act), _conv(hid, hid, 3, stride=stride, act=act, groups=hid, op="dwconv", src=0),
              _conv(hid, cout, 1, act="none", src=1, res_src=-1 if stride == 1 and cin == cout else -2)]
    sess, xd, ref = _mk(layers, "mb", n, h, w, cin)
    for s in (B.device_sm_count(), 37):
        G.check_plan(sess, xd, ref, [2], [s], "block S=%d" % s)
        name, grid, _ = sess.launches()[0]
        assert name == "mbconv_tc_kernel<%d, %s>" % (stride, "true" if act == "relu6" else "false") and 2 < grid <= s, (name, grid)
    sess.close()
