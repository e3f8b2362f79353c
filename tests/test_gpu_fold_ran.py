"""Which passes a folded query's points went through: its own FP64 form settles every tie, so
that nothing reaches the general passes, which the same query takes with folding off."""
import numpy as np
import pytest

import oracle
import synth
from gpu_common import compare, run_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    import paper_1907_12933_gb300 as m
    from paper_1907_12933_gb300 import build
    build.build()
    return m


@pytest.mark.parametrize("dims,s,k,prec", [
    ([40, 33, 5], 3, 6, "fp32"), ([100, 70, 50, 31], 2, 9, "fp32"), ([64, 64, 64, 10], 3, 6, "bf16"),
    ([64, 64, 64, 10], 2, 12, "fp16"), ([784, 512, 512, 10], 2, 9, "bf16"), ([784, 256, 256, 10], 2, 9, "fp8"),
])
def test_margin_ties_stay_on_the_folded_net(vb, dims, s, k, prec):
    net = synth.make_net(930, dims, "relu", 2.0, "normal")
    q = synth.make_query(930, 3, dims[0], s, k)
    D = oracle.eval_point(net, dict(q, pixels=q["pixels"][:0], k=0), 0)["D"]
    net["W"][-1][(D + 1) % dims[-1]] = net["W"][-1][D]
    net["b"][-1][(D + 1) % dims[-1]] = net["b"][-1][D]
    o = oracle.verify(net, q)
    assert o["n_ties"] > 0
    vnet = vb.Net(net)
    for on in (True, False):
        vb.set_folding(vnet, on)
        g = run_gpu(vb, net, q, prec, vbnet=vnet)
        compare(g, o, net, q)
        n = g["summary"]["n_recheck"]
        if on:
            assert n[0] >= o["n_ties"] and list(n[1:]) == [0, 0, 0]
        else:
            assert n[3] >= o["n_ties"]
    vnet.free()


def test_sign_ties_stay_on_the_folded_net(vb):
    """A hidden neuron whose potential is exactly 0 where two pixels' steps differ by 3."""
    net = synth.make_net(931, [12, 40, 34, 4], "relu", 2.0, "zero")
    q = synth.make_query(931, 2, 12, 2, 12)
    p0, p1 = (int(p) for p in q["pixels"])
    q["image"][p0], q["image"][p1] = 100, 103
    net["W"][0][5] = 0.0
    net["W"][0][5, p0], net["W"][0][5, p1] = 0.5, -0.5
    o = oracle.verify(net, q)
    assert o["flip_tie"].any() and o["ss_tie"].any()
    g = run_gpu(vb, net, q, "fp32")
    compare(g, o, net, q)
    n = g["summary"]["n_recheck"]
    assert n[0] > 0 and list(n[1:]) == [0, 0, 0]
