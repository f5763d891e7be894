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
