"""Inverted-residual blocks on few images (one tile per CTA or cluster): every cluster size at both strides, hidden widths that leave the
last chunk or its last 32-channel group part empty, chunks of 64, 96 and 128 channels, one buffer of each and several, windows over every
edge of the image, a unit's rows by one, two and four warps, several units to an accumulator and several accumulators, units past the
last one, one to four input planes, outputs wider than one product, SM counts that leave no room for clusters; infinities and NaN."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_05630_b200 import binding as B, synth
from tests import gpu_util as G
from tests.test_gpu_nonfinite import check_nonfinite
from tests.test_gpu_parity import _conv, _mk

# (n, h, w, cin, hidden, cout, stride, SMs (0: all), CTAs of a cluster, activation)
CASES = [
    (1, 7, 7, 160, 960, 160, 1, 0, 8, "relu6"),      # residual
    (1, 14, 14, 64, 384, 64, 1, 0, 4, "relu6"),      # chunks of 96 channels, residual
    (2, 9, 11, 40, 240, 64, 1, 0, 2, "relu6"),       # last group of half the width
    (5, 20, 29, 72, 528, 136, 1, 0, 2, "relu6"),     # several chunks per CTA, two units to an accumulator
    (1, 28, 28, 32, 192, 32, 1, 0, 1, "relu6"),      # last chunk of two groups
    (3, 30, 29, 24, 144, 24, 1, 0, 1, "relu6"),      # last chunk of half a group
    (40, 14, 14, 64, 384, 64, 1, 0, 1, "relu6"),     # four units to an accumulator, of two images
    (1, 15, 17, 24, 144, 32, 2, 0, 2, "relu"),
    (1, 57, 50, 16, 96, 24, 2, 0, 1, "relu6"),       # a chunk of three groups
    (1, 7, 7, 160, 960, 320, 1, 0, 8, "relu6"),      # projection issued as two halves
    (3, 13, 9, 96, 160, 448, 1, 0, 1, "none"),       # the widest output
    (1, 1, 1, 8, 128, 8, 1, 0, 1, "relu6"),          # one pixel
    (1, 3, 2, 256, 1024, 16, 2, 0, 8, "relu6"),      # four input planes
    (2, 16, 16, 16, 128, 16, 1, 7, 1, "relu6"),
    (1, 8, 8, 16, 128, 16, 1, 1, 1, "relu"),
    (29, 6, 5, 16, 176, 144, 1, 20, 1, "relu6"),     # three units, an accumulator each, the last tile short of two
    (21, 27, 9, 16, 336, 24, 2, 20, 1, "relu6"),     # eight units, two to an accumulator, the last tile short of five
    (1, 6, 38, 8, 320, 32, 1, 20, 4, "none"),        # a cluster with four units to an accumulator, units past the last
    (7, 9, 5, 160, 304, 96, 2, 0, 4, "relu6"),       # the same at stride 2, three input planes
    (3, 7, 20, 16, 496, 56, 2, 20, 4, "relu"),       # a cluster with three accumulators
    (4, 14, 14, 96, 576, 160, 2, 0, 4, "relu6"),     # two chunks per CTA of a cluster
    (1, 4, 9, 160, 592, 16, 2, 0, 8, "relu"),        # ... of 64 channels
    (1, 13, 13, 256, 544, 256, 1, 20, 4, "relu6"),   # three chunks of 64 per CTA, one buffer of each, residual
    (4, 10, 37, 160, 144, 352, 2, 60, 1, "relu6"),   # the same without a cluster, projection issued as two halves
    (3, 6, 5, 136, 192, 136, 1, 60, 1, "relu6"),     # two chunks of 128 channels through one buffer
    (1, 15, 4, 96, 352, 24, 2, 20, 4, "relu6"),      # chunks of 96 channels, rows by two warps
    (19, 13, 12, 8, 304, 8, 2, 20, 1, "relu6"),      # rows by four warps, one accumulator
    (4, 112, 112, 16, 96, 24, 2, 0, 1, "relu6"),     # two units, an accumulator each, rows by two warps
    (7, 7, 7, 160, 960, 160, 1, 0, 8, "none"),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "n%d_%dx%d_%d_%d_%d_s%d_sm%d" % c[:8])
def test_block(case):
    n, h, w, cin, hid, cout, stride, sms, split, act = case
    layers = [_conv(cin, hid, 1, act=act), _conv(hid, hid, 3, stride=stride, act=act, groups=hid, op="dwconv", src=0),
              _conv(hid, cout, 1, act="none", src=1, res_src=-1 if stride == 1 and cin == cout else -2)]
    sess, xd, ref = _mk(layers, "mbl", n, h, w, cin)
    G.check_plan(sess, xd, ref, [2], [sms or B.device_sm_count()], "block")
    assert sess.launches()[0][0] == "mbconv_lat_kernel<%d, %s, %d>" % (stride, "true" if act == "relu6" else "false", split)
    assert sess.launches()[0][1] <= (sms or B.device_sm_count())
    first = sess.run(xd).clone()
    assert bool((sess.run(xd) == first).all())   # the same sum whatever the timing
    sess.close()


# (n, h, w, cin, hidden, cout, stride, SMs): room for chunks of 64 hidden channels and one buffer of each only, where the persistent kernel is
# the faster one (32 us against 37, 56 against 63, 37 against 49)
@pytest.mark.parametrize("case", [(18, 14, 14, 128, 384, 96, 2, 16), (21, 9, 5, 192, 1024, 192, 1, 16), (18, 14, 14, 192, 768, 192, 1, 37)], ids=str)
def test_wide_blocks_in_many_narrow_chunks_stay_with_the_persistent_kernel(case):
    n, h, w, cin, hid, cout, stride, sms = case
    layers = [_conv(cin, hid, 1, act="relu6"), _conv(hid, hid, 3, stride=stride, act="relu6", groups=hid, op="dwconv", src=0),
              _conv(hid, cout, 1, act="none", src=1, res_src=-1 if stride == 1 and cin == cout else -2)]
    sess, xd, ref = _mk(layers, "mbl", n, h, w, cin)
    G.check_plan(sess, xd, ref, [2], [sms], "block")
    assert sess.launches()[0][0] == "mbconv_tc_kernel<%d, true>" % stride
    sess.close()


@pytest.mark.parametrize("act", ["none", "relu", "relu6"])
@pytest.mark.parametrize("stride", [1, 2])
def test_nan_and_infinity(stride, act):
    layers = [_conv(16, 128, 1, act=act), _conv(128, 128, 3, stride=stride, act=act, groups=128, op="dwconv", src=0), _conv(128, 24, 1, act=act, src=1)]
    params = synth.layer_params("mbl nonfinite", layers)
    x = synth.network_input("mbl nonfinite", 1, 21, 19, 16)
    for i, v in enumerate((np.inf, -np.inf, np.nan)):
        x[0, (2 + 8 * i) % 21, (3 + 6 * i) % 19, i] = v
    check_nonfinite(layers, params, x, [2], 0, "mbconv_lat " + act)
