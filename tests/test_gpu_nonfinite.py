"""What becomes of infinities and NaN: they stay within the windows that read them, and an activation treats a NaN as the CPU
checker does (0 behind ReLU and ReLU6), whichever kernel the sizes of a layer send it to."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import executor as orc
from paper_2011_05630_b200 import binding as B, synth
from paper_2011_05630_b200.runtime import Session
from tests import gpu_util as G
from tests.test_gpu_parity import _conv

# (name, layers, n, h, w, group ends, SMs)
LAYERS = [
    ("narrow", lambda a: [_conv(64, 64, 1, act=a)], 8, 28, 28, [0], 0),
    ("lat", lambda a: [_conv(256, 64, 1, act=a)], 1, 14, 14, [0], 0),
    ("lat cluster", lambda a: [_conv(256, 64, 3, act=a)], 1, 7, 7, [0], 0),
    ("lat residual", lambda a: [_conv(64, 64, 3, act=a, res_src=-1)], 1, 14, 14, [0], 0),
    ("tc", lambda a: [_conv(128, 128, 3, stride=2, act=a)], 1, 28, 28, [0], 1),
    ("tc residual", lambda a: [_conv(128, 128, 3, act=a, res_src=-1)], 1, 26, 28, [0], 3),
    ("tc pairs", lambda a: [_conv(128, 128, 3, act=a)], 1, 26, 28, [0], 4),
    ("chain", lambda a: [_conv(16, 16, 3, act=a), _conv(16, 16, 3, act=a, src=0)], 2, 20, 21, [1], 0),
    ("stem", lambda a: [_conv(3, 32, 4, act=a)], 1, 19, 22, [0], 0),
    ("dw", lambda a: [_conv(32, 32, 3, act=a, groups=32, op="dwconv")], 2, 15, 14, [0], 0),
    ("mbconv", lambda a: [_conv(16, 96, 1, act=a), _conv(96, 96, 3, act=a, groups=96, op="dwconv", src=0), _conv(96, 16, 1, act=a, src=1)], 1, 14, 13, [2], 0),
]


def check_nonfinite(layers, params, x, ends, sms, what):
    with np.errstate(all="ignore"):
        ref = orc.run_network(layers, params, x)[-1].astype(np.float64)
    n, h, w, c = x.shape
    s = Session(layers, params, n, h, w, c)
    s.set_plan(ends, [sms or B.device_sm_count()] * len(ends))
    got = s.run(s.upload(x)).cpu().numpy().astype(np.float64)
    s.close()
    assert not np.isfinite(ref).all() or "relu" in what   # (the values got there)
    assert (np.isnan(got) == np.isnan(ref)).all(), (what, int(np.isnan(got).sum()), int(np.isnan(ref).sum()))
    inf = np.isinf(ref)
    assert (np.isinf(got) == inf).all() and (got[inf] == ref[inf]).all(), what
    ok = np.isfinite(ref)
    assert (np.abs(got[ok] - ref[ok]) <= G.TOL * (1 + np.abs(ref[ok]))).all(), what


@pytest.mark.parametrize("act", ["none", "relu", "relu6"])
@pytest.mark.parametrize("case", LAYERS, ids=lambda c: c[0].replace(" ", "_"))
def test_nan_and_infinity(case, act):
    name, layers, n, h, w, ends, sms = case
    layers = layers(act)
    params = synth.layer_params("nonfinite", layers)
    x = synth.network_input("nonfinite", n, h, w, layers[0]["cin"])
    for i, v in enumerate((np.inf, -np.inf, np.nan)):
        x[n - 1, (2 + 5 * i) % h, (3 + 4 * i) % w, i] = v
    check_nonfinite(layers, params, x, ends, sms, name + " " + act)


# kernel widths that leave columns of a K step over: the pixels beside a window are read and must not count
@pytest.mark.parametrize("cin,cout,k,stride,pad,n,h,w", [
    (3, 64, 7, 2, 3, 2, 45, 50), (3, 32, 3, 2, 1, 1, 37, 41), (3, 64, 11, 4, 2, 1, 67, 71), (3, 64, 3, 1, 1, 1, 20, 35), (1, 16, 5, 2, 2, 1, 24, 40),
    (2, 40, 1, 1, 0, 1, 19, 21), (4, 24, 9, 4, 4, 1, 40, 41), (3, 8, 5, 1, 0, 1, 17, 33)])
def test_stem_keeps_them_in_their_windows(cin, cout, k, stride, pad, n, h, w):
    for act in ("none", "relu6"):
        layers = [_conv(cin, cout, k, stride=stride, pad=pad, act=act)]
        params = synth.layer_params("nonfinite stem", layers)
        x = synth.network_input("nonfinite stem", n, h, w, cin)
        for i, v in enumerate((np.inf, -np.inf, np.nan, np.inf)):
            x[n - 1, (3 + 4 * i) % h, (5 + 7 * i) % w, i % cin] = v
        x[n - 1, 0, 0, 0], x[0, h - 1, w - 1, cin - 1] = np.inf, np.nan
        check_nonfinite(layers, params, x, [0], 0, "stem " + ("relu6" if act == "relu6" else ""))
