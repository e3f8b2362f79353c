"""Folded nets at the limits of their number formats and of the queues behind them."""
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


def large_net(dims, scale):
    """Hidden weights of about 10^scale[l], an output layer that brings them back to 1."""
    net = synth.make_net(840, dims, "relu", 2.0, "zero")
    for l, e in enumerate(scale):
        net["W"][l] = (net["W"][l] * np.float32(10.0 ** e)).astype(np.float32)
    return net


def near_query(net, seed, h0, s, k):
    """Of 300 images, the one with the smallest margin in proportion to its largest output."""
    def closeness(q):
        o = oracle.eval_point(net, dict(q, pixels=q["pixels"][:0], k=0), 0)
        return abs(o["margin"]) / np.abs(o["u"][-net["dims"][-1]:]).max()
    return min((synth.make_query(seed, i, h0, s, k) for i in range(300)), key=closeness)


# dims, exponents of the hidden layers' weights, s, k. The products of two layers pass
# FP32's 3.4e38; FP64 holds every potential. (The tensor paths refuse such weights.)
LARGE = [
    ([12, 40, 36, 4], (20, 20), 2, 120),
    ([12, 40, 48, 40, 4], (13, 13, 13), 2, 90),
    ([12, 40, 36, 4], (37, 30), 3, 20),
    ([12, 40, 36, 4], (19, 19), 3, 20),     # products near the format's end
    ([12, 40, 36, 4], (20, 20), 1, 0),      # a box of one point: changes of 0
    ([12, 40, 36, 4], (-20, -25), 2, 9),    # products below the smallest FP32 number
]


@pytest.mark.parametrize("dims,scale,s,k", LARGE)
@pytest.mark.parametrize("coverage", [True, False])
def test_rows_past_fp32(vb, dims, scale, s, k, coverage):
    net = large_net(dims, scale)
    q = near_query(net, 840, 12, s, k)
    o = oracle.verify(net, q, coverage=coverage)
    assert 0 < o["n_adv"] < o["n_points"] or k < 10
    compare(run_gpu(vb, net, q, "fp32", coverage=coverage), o, net, q, coverage=coverage)


@pytest.mark.parametrize("d", [2e38, 3.3e38])
def test_margins_past_fp32(vb, d):
    """Output rows whose difference no FP32 number holds."""
    net = synth.make_net(841, [12, 40, 36, 4], "relu", 2.0, "normal")
    net["W"][2] = np.where(net["W"][2] < 0, -d, d).astype(np.float32)
    q = near_query(net, 841, 12, 2, 60)
    o = oracle.verify(net, q)
    assert 0 < o["n_adv"] < o["n_points"]
    compare(run_gpu(vb, net, q, "fp32"), o, net, q)


@pytest.mark.parametrize("graph", [False, True])
def test_batch_with_rows_past_fp32(vb, graph):
    net = large_net([12, 40, 36, 4], (20, 20))
    qs = [dict(near_query(net, 840, 12, 1 + i % 3, [90, 120, 20][i % 3])) for i in range(5)]
    vnet = vb.Net(net)
    res = vb.result_create_batch(vnet, len(qs), max_points=1 << 17, max_s=3, max_k=120, queue_cap=1 << 18)
    for q, r, s in zip(qs, res, vb.verify_batch(vnet, res, qs, precision="fp32", bitmap=True, graph=graph)):
        n = oracle.space_size(len(q["pixels"]), q["k"])
        compare({"summary": s, "n": n, "bitmap": vb.get_verdict_bitmap(r, n), "ties": np.sort(vb.get_ties(r)),
                 "witness": vb.get_witness(r, len(q["pixels"]), 12), **vb.get_coverage(r)},
                oracle.verify(net, q), net, q)
    for r in res:
        r.free()
    vnet.free()
