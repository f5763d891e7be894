"""Global average pooling: channel counts around a block's 64 channels, one pixel, pixels around the 32 shares, many images."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_05630_b200 import binding as B
from tests import gpu_util as G
from tests.test_gpu_parity import _mk


@pytest.mark.parametrize("n,h,w,c", [(1, 7, 7, 2048), (3, 1, 1, 8), (2, 31, 1, 72), (2, 4, 8, 64), (5, 3, 11, 136), (300, 2, 3, 128)])
def test_gavgpool(n, h, w, c):
    layer = dict(op="gavgpool", act="none", cin=c, cout=c, kh=1, kw=1, stride=1, pad=0, groups=1, src=-1, res_src=-2, pool=0)
    sess, xd, ref = _mk([layer], "gavg", n, h, w, c)
    for s in (B.device_sm_count(), 3):
        G.check_plan(sess, xd, ref, [0], [s], "gavgpool S=%d" % s)
    sess.close()
