"""Layers small enough for one output tile per CTA (conv_lat.cu): K shared out over clusters of 1, 2, 4 and 8 CTAs, rows that do
not divide by the cluster, rings that go round, ragged tiles and channel counts, residuals, a second source."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_05630_b200 import binding as B
from tests import gpu_util as G
from tests.test_gpu_parity import _conv, _mk

# (n, h, w, cin, cout, k, stride, act)
CASES = [
    (1, 56, 56, 64, 64, 1, 1, "relu"),        # a list of pixels, no split
    (1, 7, 7, 512, 512, 3, 1, "none"),        # 49 rows, 72 chunks over eight CTAs: rows 7 per CTA
    (1, 14, 14, 256, 264, 3, 2, "relu6"),     # strided taps, a last channel tile of 8
    (2, 9, 11, 24, 40, 3, 1, "relu"),         # one partial chunk per tap (24 of 64 channels), 48-wide channel tile
    (1, 5, 7, 96, 16, 5, 1, "relu"),          # 50 chunks, narrowest channel tile
    (5, 27, 29, 64, 64, 3, 1, "relu"),        # many small tiles
    (3, 1, 1, 2048, 1000, 1, 1, "none"),      # 1x1 images
    (1, 13, 13, 136, 72, 3, 1, "relu"),       # last chunk of 8 channels
    (9, 6, 6, 192, 128, 3, 2, "relu"),        # several images per tile
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "n%d_%dx%d_%d_%d_k%d_s%d" % c[:7])
def test_small_layer(case):
    n, h, w, cin, cout, k, stride, act = case
    sess, xd, ref = _mk([_conv(cin, cout, k, stride=stride, act=act)], "small", n, h, w, cin)
    sms = B.device_sm_count()
    for s in (sms, 70, 40, 20, sms):    # fewer SMs: smaller clusters, larger tiles, in the end the persistent kernel
        G.check_plan(sess, xd, ref, [0], [s], "small S=%d" % s)
    sess.close()


@pytest.mark.parametrize("n,h,w", [(1, 14, 14), (2, 9, 7)])
def test_small_block_with_residual_and_projection(n, h, w):
    """Reduce, 3x3 with stride, projection + expansion as one product, then an identity block's 3x3 layer with a residual."""
    layers = [_conv(128, 64, 1, src=-1), _conv(64, 64, 3, stride=2, src=0), _conv(128, 256, 1, stride=2, pad=0, act="none", src=-1),
              _conv(64, 256, 1, src=1, res_src=2), _conv(256, 256, 3, src=3, res_src=3)]
    sess, xd, ref = _mk(layers, "smallblock", n, h, w, 128)
    sms = B.device_sm_count()
    for ends in ([0, 1, 2, 3, 4], [0, 1, 3, 4]):
        G.check_plan(sess, xd, ref, ends, [sms] * len(ends), "block %s" % ends)
    sess.close()
