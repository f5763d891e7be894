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
