"""First-layer convolutions (at most four input channels): the tensor-core kernel reads its operand straight out of the staged
input patch, in a layout that depends on the stride.  Sizes at the edges of its 8 x 16 output tiles and of its patch: one pixel
more and less than a tile, maps smaller than a tile, several tiles per work item, tensors with an odd number of elements (the
last 32-bit word holds one), kernels that fill a K step and ones that do not, every channel count, every stride."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_05630_b200 import binding as B
from tests import gpu_util as G
from tests.test_gpu_parity import _conv, _mk

# (n, h, w, cin, cout, k, stride, pad, act)
CASES = [
    (2, 33, 35, 3, 32, 3, 2, 1, "relu6"),
    (1, 63, 67, 3, 64, 7, 2, 3, "relu"),      # odd number of input elements, 32 x 34 outputs
    (3, 15, 17, 3, 64, 3, 1, 1, "none"),      # one row short of a tile, two tiles and a column
    (1, 5, 7, 3, 8, 3, 1, 0, "relu"),         # smaller than one tile, no padding
    (2, 67, 63, 3, 64, 11, 4, 2, "relu"),     # two planes of units, 16 x 15 outputs
    (1, 227, 230, 3, 64, 11, 4, 2, "relu"),
    (2, 24, 40, 1, 16, 5, 2, 2, "none"),
    (2, 19, 21, 2, 40, 4, 1, 1, "relu6"),     # even kernel, channels that are no multiple of 16
    (1, 40, 41, 4, 64, 9, 4, 4, "relu"),
    (2, 30, 66, 3, 48, 1, 2, 0, "none"),      # 1x1
    (150, 9, 9, 3, 24, 3, 1, 1, "relu"),      # more work items than SMs
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "n%d_%dx%d_%d_%d_k%d_s%d_p%d" % c[:8])
def test_stem(case):
    n, h, w, cin, cout, k, stride, pad, act = case
    layer = _conv(cin, cout, k, stride=stride, pad=pad, act=act)
    sess, xd, ref = _mk([layer], "stem", n, h, w, cin)
    for s in (B.device_sm_count(), 5):
        G.check_plan(sess, xd, ref, [0], [s], "stem S=%d" % s)
        assert sess.kernels() == ["stem_tc"]
    sess.close()
