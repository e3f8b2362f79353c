"""The witness of a query whose inputs lay in device memory that has since been given to
others: its image, steps and margin are those of the inputs at the call."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1907_12933_gb300 as m
    from paper_1907_12933_gb300 import build
    build.build()
    return m


@pytest.mark.parametrize("dims,act,prec", [([30, 40, 20, 4], "relu", "fp32"), ([25, 10, 5], "sigmoid", "fp64"),
                                           ([700, 64, 64, 6], "relu", "bf16")])
@pytest.mark.parametrize("member", [False, True])
def test_witness_of_device_inputs(vb, dims, act, prec, member):
    import torch
    net = synth.make_net(880, dims, act, 2.0, "normal")
    q = synth.make_query(880, 2, dims[0], 3, 12)
    y = oracle.eval_point(net, dict(q, pixels=q["pixels"][:0], k=0), 0)["u"][-dims[-1]:]
    net["b"][-1] += (0.002 * np.arange(dims[-1]) - y).astype(np.float32)
    o = oracle.verify(net, q)
    assert o["first_witness"] is not None
    n = oracle.space_size(3, 12)
    vnet = vb.Net(net)
    kw = {"max_points": n, "max_s": 3, "max_k": 12, "queue_cap": n}
    res = vb.result_create_batch(vnet, 2, **kw) if member else [vb.Result(vnet, **kw)]
    other = dict(q, image=255 - np.asarray(q["image"]))
    if member:  # the handle's last call had another image
        vb.verify_batch(vnet, res, [other, other], precision=prec)
    else:
        vb.verify_query(vnet, res[0], other["image"], other["pixels"], 12, precision=prec)
    img = torch.from_numpy(np.asarray(q["image"], np.uint8)).cuda()
    pix = torch.from_numpy(np.asarray(q["pixels"], np.int32)).cuda()
    vb.verify_query_device(vnet, res[0], img, pix, 12, precision=prec)
    img.fill_(7)
    pix.fill_(1)
    s = vb.result_summary(res[0])
    compare({"summary": s, "n": n, "bitmap": vb.get_verdict_bitmap(res[0], n), "ties": np.sort(vb.get_ties(res[0])),
             "witness": vb.get_witness(res[0], 3, dims[0]), **vb.get_coverage(res[0])}, o, net, q)
    for r in res:
        r.free()
    vnet.free()
