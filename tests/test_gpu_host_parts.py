"""dlf_net_run_host on batches large enough to be worked off in parts while the input arrives: ragged parts, every kind of
group that may lead a plan, the same output as a run on device memory, again after new plans and new inputs."""
import numpy as np
import pytest
import torch

from paper_2011_05630_b200 import binding as B
from paper_2011_05630_b200 import networks as nw
from paper_2011_05630_b200 import plans
from paper_2011_05630_b200.runtime import Session

pytestmark = pytest.mark.gpu


def _chain():
    return nw.conv_chain(3, 16, 3) + [dict(l, src=l["src"] + 3) for l in nw.conv_chain(2, 16, 1)]


@pytest.mark.parametrize("layers,n,h,w,c", [
    (nw.resnet50(), 29, 224, 224, 3), (nw.mobilenet_v2(), 31, 200, 232, 3), (nw.resnet18(), 33, 211, 224, 3), (_chain(), 19, 128, 120, 16)])
def test_parts_of_a_batch(layers, n, h, w, c):
    g = torch.Generator().manual_seed(n)
    params = []
    for l in layers:
        if l["op"] in ("conv", "dwconv"):
            shape = (l["cout"], l["kh"], l["kw"], l["cin"] // l["groups"])
        elif l["op"] == "fc":
            shape = (l["cout"], l["cin"])
        else:
            params.append(None)
            continue
        fan = int(np.prod(shape[1:]))
        params.append(((torch.randn(shape, generator=g) * fan ** -0.5).half().numpy(), (torch.randn(l["cout"], generator=g) * 0.1).numpy()))
    s = Session(layers, params, n, h, w, c)
    assert n * h * w * c * 2 >= 8 << 20   # (the copy is long enough to be cut)
    y = torch.empty(s.out_shape, dtype=torch.float16, pin_memory=True)
    stream = torch.cuda.current_stream().cuda_stream
    for tuned in (False, True):
        s.set_plan(*plans.tuned_plan(s.net, len(layers))) if tuned else s.set_plan()
        for seed in (1, 2):
            x = (torch.rand((n, h, w, c), generator=torch.Generator().manual_seed(seed)) * 2 - 1).half().pin_memory()
            y.fill_(float("nan"))
            B.net_run_host(s.net, x.data_ptr(), y.data_ptr(), stream)
            ref = s.run(x.cuda()).float().cpu()
            # a part may run through other tiles: sums in another order, single fp16 roundings carried on through the layers
            assert float((y.float() - ref).norm() / ref.norm()) < 2e-3
    s.close()


@pytest.mark.parametrize("n,h,w", [(27, 203, 261), (29, 203, 261), (30, 203, 261), (19, 287, 287)])
def test_parts_of_images_with_an_odd_number_of_elements(n, h, w):
    """An image of 2 mod 4 bytes: a part may not start on an odd one, whatever the quarters of the batch come to."""
    layers = nw.resnet18()
    assert h * w * 3 % 2 == 1 and n * h * w * 3 * 2 >= 8 << 20
    g = torch.Generator(device="cuda").manual_seed(n)
    params = []
    for l in layers:
        if l["op"] not in ("conv", "fc"):
            params.append(None)
            continue
        shape = (l["cout"], l["kh"], l["kw"], l["cin"]) if l["op"] == "conv" else (l["cout"], l["cin"])
        params.append(((torch.randn(shape, generator=g, device="cuda") * int(np.prod(shape[1:])) ** -0.5).half().cpu().numpy(),
                       (torch.randn(l["cout"], generator=g, device="cuda") * 0.1).cpu().numpy()))
    s = Session(layers, params, n, h, w, 3)
    s.set_plan(*plans.tuned_plan(s.net, len(layers)))
    x = (torch.rand((n, h, w, 3), generator=g, device="cuda") * 2 - 1).half()
    ref = s.run(x).float().cpu()
    xh, y = x.cpu().pin_memory(), torch.empty(s.out_shape, dtype=torch.float16, pin_memory=True)
    B.net_run_host(s.net, xh.data_ptr(), y.data_ptr(), torch.cuda.current_stream().cuda_stream)
    s.close()
    # single fp16 roundings (see above)
    assert float((y.float() - ref).norm() / ref.norm()) < 2e-3


def test_parts_from_pageable_memory():
    """Buffers that are not page-locked, overwritten as soon as the call is back."""
    layers = _chain()
    g = torch.Generator().manual_seed(7)
    params = [((torch.randn((l["cout"], l["kh"], l["kw"], l["cin"]), generator=g) * (l["kh"] * l["kw"] * l["cin"]) ** -0.5).half().numpy(),
               (torch.randn(l["cout"], generator=g) * 0.1).numpy()) for l in layers]
    s = Session(layers, params, 20, 128, 120, 16)
    s.set_plan(*plans.tuned_plan(s.net, len(layers)))
    x = (torch.rand((20, 128, 120, 16), generator=g) * 2 - 1).half()
    y = torch.empty(s.out_shape, dtype=torch.float16)
    for _ in range(3):
        xh = x.clone()
        y.fill_(float("nan"))
        B.net_run_host(s.net, xh.data_ptr(), y.data_ptr(), torch.cuda.current_stream().cuda_stream)
        xh.fill_(float("nan"))
        ref = s.run(x.cuda()).float().cpu()
        assert float((y.float() - ref).norm() / ref.norm()) < 2e-3   # (see above)
        x = -x
    s.close()
