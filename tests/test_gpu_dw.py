"""Depthwise 3x3: strips of one row up to the whole column, the three-row ring's remainders, columns at the image's edges, maps
smaller than the kernel, both strides, channel counts whose quarter is odd, residuals."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_05630_b200 import binding as B
from tests import gpu_util as G
from tests.test_gpu_parity import _conv, _mk

CASES = [(1, 14, 14, 384, 1), (1, 1, 1, 8, 1), (2, 2, 3, 24, 2), (1, 5, 1, 40, 1), (3, 17, 19, 72, 2), (2, 40, 9, 16, 1), (1, 64, 33, 32, 2),
         (30, 23, 21, 24, 1)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "n%d_%dx%d_%d_s%d" % c)
def test_dw(case):
    n, h, w, c, stride = case
    sess, xd, ref = _mk([_conv(c, c, 3, stride=stride, act="relu6", groups=c, op="dwconv")], "dw", n, h, w, c)
    for s in (B.device_sm_count(), 3, 1):   # fewer SMs: longer strips, more rounds
        G.check_plan(sess, xd, ref, [0], [s], "dw S=%d" % s)
        assert sess.kernels() == ["dw3x3"]
    sess.close()


def test_dw_with_residual():
    layers = [_conv(16, 16, 3, act="none", groups=16, op="dwconv"), _conv(16, 16, 3, groups=16, op="dwconv", src=0, res_src=-1)]
    sess, xd, ref = _mk(layers, "dwres", 2, 11, 13, 16)
    G.check_plan(sess, xd, ref, [0, 1], [B.device_sm_count()] * 2, "dw residual")
    sess.close()
