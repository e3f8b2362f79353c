"""The FP64 pass over a filtered range: many points per CTA, most of them, some of them and
none of them skipped, against the oracle."""
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


@pytest.mark.parametrize("dims,act", [([25, 10, 5], "sigmoid"), ([30, 40, 20, 4], "relu"), ([20, 300, 3], "identity")])
@pytest.mark.parametrize("filt,l2", [(1, 40), (1, 120), (1, 1 << 20), (2, 0), (3, 150)])
def test_filtered_range(vb, dims, act, filt, l2):
    net = synth.make_net(850, dims, act, 2.0, "normal")
    q = synth.make_query(850, 2, dims[0], 4, 8)
    y = oracle.eval_point(net, dict(q, pixels=q["pixels"][:0], k=0), 0)["u"][-dims[-1]:]
    net["b"][-1] += (0.002 * np.arange(dims[-1]) - y).astype(np.float32)
    n = oracle.space_size(4, 8)
    vnet = vb.Net(net)
    res = vb.Result(vnet, max_points=n, max_s=4, max_k=8)
    o = oracle.verify(net, dict(q, filter=filt, l2_max=l2))
    assert o["n_adv"] > 0 and o["n_points"] > 0
    for _ in range(3):
        s = vb.verify_query(vnet, res, q["image"], q["pixels"], 8, precision="fp64", filter=filt, l2_max=l2)
        compare({"summary": s, "n": n, "bitmap": vb.get_verdict_bitmap(res, n), "ties": np.sort(vb.get_ties(res)),
                 "witness": vb.get_witness(res, 4, dims[0]), **vb.get_coverage(res)}, o, net, q)
    res.free()
    vnet.free()
