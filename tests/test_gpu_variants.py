"""Which kernel a layer's size and SM count send it to, and what that kernel makes of it: every variant of the single-layer
convolution kernels is asked for by name, so that an estimate that moves cannot leave one of them untested."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_05630_b200 import binding as B
from tests import gpu_util as G
from tests import test_gpu_parity as TP
from tests.test_gpu_parity import _conv, _mk

ALL = 0   # all SMs
# (kernel, layer, n, h, w, SMs)
CASES = [
    # pointwise layers of at most 64 input channels: one and two blocks of them, partial ones, one to four eights of output channels
    ("conv_narrow_kernel<1, 1, 0, 8>", _conv(8, 8, 1, act="none"), 1, 1, 1, ALL),
    ("conv_narrow_kernel<1, 2, 2, 8>", _conv(24, 16, 1, act="relu6"), 3, 17, 13, ALL),
    ("conv_narrow_kernel<1, 3, 1, 8>", _conv(24, 24, 1, res_src=-1), 5, 31, 29, ALL),
    ("conv_narrow_kernel<1, 4, 2, 8>", _conv(16, 96, 1, act="relu6"), 4, 56, 57, ALL),
    ("conv_narrow_kernel<2, 1, 1, 8>", _conv(64, 8, 1), 2, 61, 59, ALL),
    ("conv_narrow_kernel<2, 2, 0, 8>", _conv(40, 16, 1, act="none"), 2, 61, 59, ALL),
    ("conv_narrow_kernel<2, 3, 1, 8>", _conv(48, 24, 1), 2, 61, 59, ALL),
    ("conv_narrow_kernel<2, 4, 1, 8>", _conv(56, 192, 1), 2, 61, 59, ALL),
    ("conv_narrow_kernel<2, 4, 1, 8>", _conv(64, 64, 1, res_src=-1), 7, 28, 28, ALL),
    # one tile per CTA, K over clusters of 1 to 8
    ("conv_lat_kernel<1>", _conv(64, 64, 1), 1, 56, 56, ALL),
    ("conv_lat_kernel<1>", _conv(64, 64, 3, res_src=-1), 5, 27, 29, ALL),
    ("conv_lat_kernel<2>", _conv(24, 40, 3), 2, 9, 11, ALL),
    ("conv_lat_kernel<2>", _conv(2048, 1000, 1, act="none"), 3, 1, 1, 20),
    ("conv_lat_kernel<4>", _conv(136, 72, 3), 1, 13, 13, ALL),
    ("conv_lat_kernel<4>", _conv(192, 192, 3, act="relu6", res_src=-1), 1, 14, 14, 40),
    ("conv_lat_kernel<8>", _conv(512, 512, 3, act="none"), 1, 7, 7, ALL),
    ("conv_lat_kernel<8>", _conv(96, 16, 5), 1, 5, 7, 20),
    # persistent, one CTA to a work item
    ("conv_tc_kernel<1, false, false, false, false>", _conv(72, 64, 1), 1, 20, 23, 2),
    ("conv_tc_kernel<1, false, true, true, false> by rows", _conv(64, 64, 3, res_src=-1), 1, 20, 23, 2),
    ("conv_tc_kernel<1, false, false, true, false> by columns", _conv(64, 128, 3), 1, 20, 23, 3),
    ("conv_tc_kernel<1, true, true, true, false> by columns", _conv(64, 64, 3, pool=2, res_src=-1), 1, 20, 23, 2),
    ("conv_tc_kernel<1, false, false, true, true> by rows", _conv(1024, 16, 3), 1, 14, 14, 4),    # K shared out between CTAs
    ("conv_tc_kernel<1, false, true, false, false>", _conv(64, 64, 1, res_src=-1), 16, 56, 56, ALL),   # (without a residual: conv_narrow)
    ("conv_narrow_kernel<2, 4, 1, 8>", _conv(64, 64, 1), 16, 56, 56, ALL),
    # ... two: pixel lists, strides, partial last chunks, pooling, odd SM counts (the last SM stays out)
    ("conv_tc_pair_kernel<1, false, false, false>", _conv(512, 192, 1), 1, 20, 23, 3),
    ("conv_tc_pair_kernel<1, false, true, false>", _conv(512, 512, 1, res_src=-1), 1, 20, 23, 7),
    ("conv_tc_pair_kernel<1, true, true, false>", _conv(512, 512, 1, pool=2, res_src=-1), 1, 20, 23, 5),
    ("conv_tc_pair_kernel<0, false, false, false>", _conv(512, 64, 1, stride=2, pad=0, act="none"), 1, 61, 59, 2),
    ("conv_tc_pair_kernel<1, false, false, false>", _conv(72, 192, 3), 2, 33, 31, 2),
    ("conv_tc_pair_kernel<2, true, false, false>", _conv(200, 320, 3, pool=2, act="relu6"), 1, 20, 23, 5),
    ("conv_tc_pair_kernel<1, false, true, true> by rows", _conv(64, 64, 3, res_src=-1), 1, 61, 59, 5),
    ("conv_tc_pair_kernel<1, false, false, true> by rows", _conv(64, 192, 3), 1, 20, 23, 2),
    ("conv_tc_pair_kernel<1, false, false, true> by columns", _conv(64, 128, 3), 2, 33, 31, 7),
    ("conv_tc_pair_kernel<1, false, true, true> by columns", _conv(64, 64, 3, res_src=-1), 2, 33, 31, 2),
    ("conv_tc_pair_kernel<1, true, true, true> by columns", _conv(64, 64, 3, pool=2, res_src=-1), 3, 28, 28, 7),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "%s-%d-%d-k%d-S%d" % (c[0].replace("_kernel", "").replace(" ", ""), c[1]["cin"], c[1]["cout"], c[1]["kh"], c[5]))
def test_variant(case):
    kernel, layer, n, h, w, sms = case
    sess, xd, ref = _mk([layer], "variant", n, h, w, layer["cin"])
    sms = sms or B.device_sm_count()
    G.check_plan(sess, xd, ref, [0], [sms], kernel)
    name, grid, _ = sess.launches()[0]
    sess.close()
    assert name == kernel
    if not name.startswith("conv_narrow"):
        assert grid <= sms


@pytest.mark.parametrize("cin,cout,act,res", [(8, 8, "none", False), (24, 16, "relu6", False), (24, 24, "relu", True), (32, 32, "relu", False),
                                               (16, 96, "relu6", False), (32, 256, "none", False), (64, 64, "relu", True)])
def test_narrow_layers_keep_to_the_sm_count(cin, cout, act, res):
    """One CTA on each of the SMs that the plan names, whatever is free beside them."""
    sess, xd, ref = _mk([_conv(cin, cout, 1, act=act, res_src=-1 if res else -2)], "knob", 2, 61, 59, cin)
    for sms in (B.device_sm_count() - 1, 37, 2, 1):
        G.check_plan(sess, xd, ref, [0], [sms], "narrow S=%d" % sms)
        name, grid, _ = sess.launches()[0]
        assert grid <= sms and name.startswith("conv_narrow") == (cin <= 32), (name, grid)
    sess.close()


def test_the_query_follows_the_plan():
    layers = [_conv(16, 16, 3), _conv(16, 16, 3, src=0)]
    sess, _, _ = _mk(layers, "query", 1, 32, 32, 16)
    sess.set_plan([0, 1], [20, 20])
    assert [a[0].split("<")[0] for a in sess.launches()] == ["conv_lat_kernel"] * 2
    sess.set_plan([1], [8])
    assert sess.launches()[0][0].startswith("chain_tc_kernel") and sess.launches()[0][1] == 8
    with pytest.raises(B.DlfError):
        B.net_group_launch(sess.net, 1)
    sess.close()


@pytest.mark.parametrize("kernel,layers,ends", [
    ("conv_seq_kernel", [_conv(128, 128, 3, stride=2), _conv(128, 64, 1, src=0)], [1]),
    ("dw3x3_kernel<2>", [_conv(16, 16, 3, stride=2, groups=16, op="dwconv")], [0]),
    ("maxpool_kernel", [dict(_conv(16, 16, 3, stride=2, act="none"), op="maxpool")], [0]),
    ("gavgpool_kernel", [dict(_conv(16, 16, 1, act="none"), op="gavgpool")], [0]),
    ("conv_direct_kernel", [_conv(6, 16, 3)], [0]),
    ("mbconv_tc_kernel<1, true>", [_conv(16, 96, 1, act="relu6"), _conv(96, 96, 3, groups=96, op="dwconv", act="relu6", src=0), _conv(96, 16, 1, src=1, act="none")], [2]),
], ids=lambda v: v if isinstance(v, str) else None)
def test_names_of_the_other_kernels(kernel, layers, ends):
    sess, xd, ref = _mk(layers, "names", 1, 20, 20, layers[0]["cin"])
    G.check_plan(sess, xd, ref, ends, [B.device_sm_count()] * len(ends), kernel)
    assert [a[0] for a in sess.launches()] == [kernel]
    sess.close()


def test_row_mode_option():
    """2: by rows wherever that applies, pairs or not; 0: neither by rows nor by columns."""
    for n, h, w, layer in TP.ROW_MODE:
        sess, xd, ref = _mk([layer], "rowmode", n, h, w, layer["cin"])
        try:
            for mode in (2, 0):
                B.net_set_option(sess.net, B.OPT_CONV_ROW_MODE, mode)
                for sms in (B.device_sm_count(), 5):
                    G.check_plan(sess, xd, ref, [0], [sms], "row mode %d S=%d" % (mode, sms))
                    name = sess.launches()[0][0]
                    assert name.endswith(" by rows") == (mode == 2 and w <= 126), (mode, w, name)
                    assert mode == 2 or "columns" not in name, (mode, w, name)
        finally:
            B.net_set_option(sess.net, B.OPT_CONV_ROW_MODE, 1)
        sess.close()


def test_split_reduction_over_a_pixel_list():
    """A fully connected layer of many images and a long K on few SMs: the variant of the persistent kernel that shares K out."""
    n, k, m = 200, 25088, 1000
    layers = [dict(_conv(k, m, 1), op="fc")]
    g = torch.Generator(device="cuda").manual_seed(1)
    w = (torch.randn((m, k), generator=g, device="cuda") * k ** -0.5).half()
    b = torch.randn((m,), generator=g, device="cuda") * 0.1
    x = (torch.rand((n, 1, 1, k), generator=g, device="cuda") * 2 - 1).half()
    sess = TP.Session(layers, [(w.cpu().numpy(), b.cpu().numpy())], n, 1, 1, k)
    sess.set_plan([0], [20])
    assert sess.launches()[0][0] == "conv_tc_kernel<1, false, false, false, true>"
    ref = (x.reshape(n, k).double() @ w.double().T + b.double()).clamp(min=0)
    for _ in range(2):   # (the arrival counters are back at zero after a launch)
        got = sess.run(x).reshape(n, m).double()
        # one rounding to fp16, and 25088 fp32 additions to partial sums below 8: 25088 * 8 * 2^-24 / 2 = 0.006 at the very worst,
        # its square root's share (1e-4) as a rule
        assert bool(((got - ref).abs() <= 2 ** -11 * ref + 1e-3).all())
    sess.close()
