"""Layers whose work items are shared by CTA pairs (two pixel tiles, half of the weight slab in either CTA): odd numbers of
tiles (the last pair's second tile lies past the batch), several rounds, an odd SM count, one pair, row mode, strides,
residuals, fused pooling, channel tiles that are not full, the projection + expansion product."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests import gpu_util as G
from tests.test_gpu_parity import _conv, _mk

# (n, h, w, layer)
CASES = [
    (3, 14, 14, _conv(256, 256, 3)),                    # row mode
    (5, 14, 14, _conv(128, 320, 3, act="none")),        # three or more channel tiles, the last one partial
    (2, 33, 31, _conv(192, 128, 3, stride=2)),          # window load per tap
    (3, 28, 28, _conv(256, 256, 3, pool=2)),            # pooled
    (7, 17, 19, _conv(64, 512, 1)),                     # a list of pixels
    (2, 20, 23, _conv(192, 192, 5, act="relu6")),       # 25 taps
    (3, 28, 28, _conv(512, 256, 1, stride=2, pad=0)),
    (4, 13, 13, _conv(136, 72, 3)),                     # partial last chunk
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "n%d_%dx%d_%d_%d_k%d_s%d_p%d" % (c[:3] + tuple(c[3][k] for k in ("cin", "cout", "kh", "stride", "pool"))))
def test_pairs(case):
    n, h, w, layer = case
    sess, xd, ref = _mk([layer], "pairs", n, h, w, layer["cin"])
    for s in (2, 3, 6, 2):
        G.check_plan(sess, xd, ref, [0], [s], "pairs S=%d" % s)
    sess.close()


def test_pairs_with_residual_and_projection():
    layers = [_conv(128, 128, 3, src=-1), _conv(128, 128, 3, src=0, res_src=-1), _conv(128, 256, 1, stride=2, pad=0, act="none", src=1),
              _conv(128, 128, 3, stride=2, src=1), _conv(128, 256, 1, src=3, res_src=2)]
    sess, xd, ref = _mk(layers, "pairblock", 3, 26, 22, 128)
    for s in (2, 4, 5):
        for ends in ([0, 1, 2, 3, 4],):
            G.check_plan(sess, xd, ref, ends, [s] * len(ends), "pair block S=%d" % s)
    sess.close()
