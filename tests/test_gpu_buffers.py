"""A plan follows the buffers it is called with: the captured kernels are given each call's input and output."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import executor as orc
from paper_2011_05630_b200 import binding as B, synth
from paper_2011_05630_b200.runtime import Session
from tests import gpu_util as G
from tests.test_gpu_parity import _conv


@pytest.mark.parametrize("graph", [1, 0])
def test_run_follows_the_callers_buffers(graph):
    """New input and output buffers from call to call, several runs enqueued before the first is waited for: every output is
    that of its own input (the first layer, a residual of the input and the last layer see the buffers)."""
    layers = [_conv(16, 16, 3), _conv(16, 16, 3, src=0), _conv(16, 16, 1, src=1, res_src=-1), _conv(16, 24, 3, src=2)]
    params = synth.layer_params("buffers", layers)
    sess = Session(layers, params, 2, 17, 19, 16)
    B.net_set_option(sess.net, B.OPT_CUDA_GRAPH, graph)
    for plan in ([0, 1, 2, 3], [1, 2, 3]):
        sess.set_plan(plan, [B.device_sm_count()] * len(plan))
        xs = [synth.network_input("buffers%d" % i, 2, 17, 19, 16) for i in range(3)]
        xd = [sess.upload(x) for x in xs]
        out = [torch.empty(sess.out_shape, dtype=torch.float16, device=sess.device) for _ in xs]
        stream = torch.cuda.current_stream().cuda_stream
        for i in (0, 1, 2, 1, 0):
            B.net_run(sess.net, xd[i].data_ptr(), out[i].data_ptr(), stream)
        B.net_sync(sess.net, stream)
        for x, o in zip(xs, out):
            G.compare(o.cpu().numpy(), orc.run_network(layers, params, x)[-1], "plan %s" % plan)
    sess.close()


KINDS = [   # (layers, image height and width, plan): one group of every kernel, alone in its plan
    ([_conv(64, 64, 1)], 28, 28, None),                                     # conv_narrow
    ([_conv(64, 64, 1, res_src=-1)], 28, 28, None),
    ([_conv(128, 64, 3)], 14, 14, None),                                    # conv_lat
    ([_conv(128, 128, 3)], 130, 130, None),                                 # conv_tc
    ([_conv(128, 128, 3, pool=2)], 28, 28, None),
    ([_conv(16, 16, 3), _conv(16, 24, 3, src=0)], 20, 20, [1]),             # chain_tc
    ([_conv(128, 128, 3, stride=2), _conv(128, 64, 1, src=0)], 20, 20, [1]),   # conv_seq
    ([_conv(16, 96, 1), _conv(96, 96, 3, groups=96, op="dwconv", src=0), _conv(96, 16, 1, src=1, act="none", res_src=-1)], 14, 14, [2]),
    ([_conv(64, 64, 3, groups=64, op="dwconv")], 14, 14, None),
    ([dict(_conv(64, 64, 3, stride=2, act="none"), op="maxpool")], 14, 14, None),
]


@pytest.mark.parametrize("graph", [1, 0])
@pytest.mark.parametrize("case", KINDS, ids=lambda c: "%s%d" % (c[0][0]["op"], c[0][0]["cin"]))
def test_misaligned_buffers_are_refused(case, graph):
    """The code comes back and nothing has run: the output keeps what it held, and the next call on proper buffers is right."""
    layers, h, w, plan = case
    params = synth.layer_params("misaligned", layers)
    x = synth.network_input("misaligned", 1, h, w, layers[0]["cin"])
    s = Session(layers, params, 1, h, w, layers[0]["cin"])
    B.net_set_option(s.net, B.OPT_CUDA_GRAPH, graph)
    s.set_plan(plan, [B.device_sm_count()]) if plan else s.set_plan()
    xd = torch.zeros(x.size + 64, dtype=torch.float16, device=s.device)
    yd = torch.full((s.out.numel() + 64,), 7.0, dtype=torch.float16, device=s.device)
    stream = torch.cuda.current_stream().cuda_stream
    for dx, dy in ((2, 0), (0, 2), (4, 0), (0, 4)):
        with pytest.raises(B.DlfError) as e:
            B.net_run(s.net, xd.data_ptr() + dx, yd.data_ptr() + dy, stream)
        assert e.value.status == B.E_INVALID_ARG
        with pytest.raises(B.DlfError) as e:
            B.net_time(s.net, xd.data_ptr() + dx, yd.data_ptr() + dy, s.n_groups, stream, warmup=0, iters=1)
        assert e.value.status == B.E_INVALID_ARG
    torch.cuda.synchronize()
    assert bool((yd == 7.0).all())
    G.compare(s.run(s.upload(x)).cpu().numpy(), orc.run_network(layers, params, x)[-1], "aligned again")
    s.close()
