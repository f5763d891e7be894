"""Fully connected layers on the CUDA cores at the edges of their batch tiles (1, 2, 4, 8 images), of K (fewer 16-byte pieces than threads,
one more than a whole pass) and of the features, with blocks that go on to a second tile (one SM)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2011_05630_b200 import binding as B
from paper_2011_05630_b200.runtime import Session


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 9])
def test_fc(n):
    g = torch.Generator(device="cuda").manual_seed(n)
    for k, m in ((8, 1), (40, 7), (2048, 1000), (2056, 9), (4096, 130)):
        w = (torch.randn((m, k), generator=g, device="cuda") * k ** -0.5).half()
        b = torch.randn((m,), generator=g, device="cuda") * 0.1
        x = (torch.rand((n, 1, 1, k), generator=g, device="cuda") * 2 - 1).half()
        layers = [dict(op="fc", act="none", cin=k, cout=m, kh=1, kw=1, stride=1, pad=0, groups=1, src=-1, res_src=-2, pool=0)]
        sess = Session(layers, [(w.cpu().numpy(), b.cpu().numpy())], n, 1, 1, k)
        ref = x.reshape(n, k).double() @ w.double().T + b.double()
        for sms in (B.device_sm_count(), 1):
            sess.set_plan([0], [sms])
            got = sess.run(x).reshape(n, m).double()
            # one rounding to fp16 (2^-11 of a value), and K fp32 additions to sums below 4: K * 4 * 2^-24 = 1e-3 at the very worst
            assert bool(((got - ref).abs() <= 2 ** -11 * ref.abs() + 1e-3).all()), (n, k, m, sms, sess.launches()[0][0])
        sess.close()


@pytest.mark.parametrize("graph", [0, 1])
def test_weights_that_the_work_before_writes(graph):
    """With a graph or without a run starts when all that its stream holds is done: the weights of one network are another one's output, while
    that one's kernel already lets the next start."""
    g = torch.Generator(device="cuda").manual_seed(3)
    k1, k2, m2 = 8192, 2048, 8
    fc = lambda k, m: [dict(op="fc", act="none", cin=k, cout=m, kh=1, kw=1, stride=1, pad=0, groups=1, src=-1, res_src=-2, pool=0)]
    w1 = (torch.randn((k2 * m2, k1), generator=g, device="cuda") * k1 ** -0.5).half()
    first = Session(fc(k1, k2 * m2), [(w1.cpu().numpy(), torch.zeros(k2 * m2).numpy())], 1, 1, 1, k1)
    second = Session(fc(k2, m2), [(torch.zeros((m2, k2)).half().numpy(), torch.zeros(m2).numpy())], 1, 1, 1, k2)
    w2 = second._keep[0]
    for s in (first, second):
        B.net_set_option(s.net, B.OPT_CUDA_GRAPH, graph)
        s.set_plan([0], [B.device_sm_count()])
    stream = torch.cuda.current_stream().cuda_stream
    for i in range(4):
        x1 = (torch.rand((1, 1, 1, k1), generator=g, device="cuda") * 2 - 1).half()
        x2 = (torch.rand((1, 1, 1, k2), generator=g, device="cuda") * 2 - 1).half()
        w2.zero_()
        torch.cuda.synchronize()
        B.net_run(first.net, x1.data_ptr(), w2.data_ptr(), stream)
        B.net_run(second.net, x2.data_ptr(), second.out.data_ptr(), stream)
        torch.cuda.synchronize()
        ref = x2.reshape(1, k2).double() @ w2.double().T
        # one rounding to fp16, and 2048 fp32 additions to sums below 64: 2048 * 64 * 2^-24 = 8e-3 at the very worst
        assert float(w2.abs().max()) > 0 and bool(((second.out.reshape(1, m2).double() - ref).abs() <= 2 ** -11 * ref.abs() + 8e-3).all()), i
    first.close(); second.close()
