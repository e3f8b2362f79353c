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


def all_undecided(seed, tie):
    """784-256-256-10 with a dead neuron (every sign of it a tie, so that no point's covers are
    certain in the first pass) or with two equal outputs (a margin tie at every point)."""
    net = synth.make_net(seed, [784, 256, 256, 10], "relu", 2.0, "normal")
    if tie == "sign":
        net["W"][0][17] = 0.0
        net["b"][0][17] = 0.0
    else:
        D = oracle.eval_point(net, synth.make_query(seed, 1, 784, 1, 0), 0)["D"]
        net["W"][2][(D + 1) % 10] = net["W"][2][D]
        net["b"][2][(D + 1) % 10] = net["b"][2][D]
    return net


def read(vb, res, s, n, dims, summary):
    return {"summary": summary, "n": n, "bitmap": vb.get_verdict_bitmap(res, n), "ties": np.sort(vb.get_ties(res)),
            "witness": vb.get_witness(res, s, dims[0]), **vb.get_coverage(res)}


# points per chunk of the wide-layer path, which drains its queues after each; capacity
@pytest.mark.parametrize("tie", ["sign", "margin"])
@pytest.mark.parametrize("s,k,chunk,cap", [(2, 30, 1024, 2048), (3, 20, 4096, 1 << 16), (2, 30, 1024, 1024),
                                             (3, 20, 256, 256), (2, 30, 128, 128)])
@pytest.mark.parametrize("call", ["host", "device"])
def test_wide_query_with_more_undecided_points_than_the_queue_holds(vb, tie, s, k, chunk, cap, call):
    net = all_undecided(843, tie)
    q = synth.make_query(843, 1, 784, s, k)
    n = oracle.space_size(s, k)
    assert n > cap
    vnet = vb.Net(net)
    vb.net_prepare(vnet, "fp8")
    res = vb.Result(vnet, max_points=n, max_s=s, max_k=k, ties_cap=1 << 17, queue_cap=cap, wide_chunk=chunk)
    o = oracle.verify(net, q, ties_cap=1 << 17)
    for _ in range(2):
        if call == "host":
            summ = vb.verify_query(vnet, res, q["image"], q["pixels"], k, precision="fp8", bitmap=True)
        else:
            import torch
            img = torch.from_numpy(np.asarray(q["image"], np.uint8)).cuda()
            pix = torch.from_numpy(np.asarray(q["pixels"], np.int32)).cuda()
            vb.verify_query_device(vnet, res, img, pix, k, precision="fp8", bitmap=True)
            summ = vb.result_summary(res)
        g = read(vb, res, s, n, net["dims"], summ)
        g["ties"] = np.sort(vb.get_ties(res, 1 << 17))
        compare(g, o, net, q)
    res.free()
    vnet.free()


def test_wide_search_and_shells_with_more_undecided_points_than_the_queue_holds(vb):
    net = all_undecided(844, "margin")
    q = synth.make_query(844, 1, 784, 2, 30)
    n = oracle.space_size(2, 30)
    vnet = vb.Net(net)
    res = vb.Result(vnet, max_s=2, max_k=30, ties_cap=1 << 13, queue_cap=512, wide_chunk=512)
    o = oracle.verify(net, q)
    assert o["n_adv"] == 0 and o["n_ties"] == n
    r = vb.search_query(vnet, res, q["image"], q["pixels"], 30, np.array([2, 0, 1]), precision="fp8")
    assert (r["n_points"], r["n_ties"], r["n_adversarial"], r["tiles_checked"]) == (n, n, 0, 3)
    sh = vb.shell_search(vnet, res, q["image"], q["pixels"], 30, precision="fp8")
    assert (sh["radius"], sh["points_checked"], sh["ties_total"]) == (None, n, n)
    res.free()
    vnet.free()


@pytest.mark.parametrize("graph", [False, True])
def test_batch_past_its_queue_is_refused_and_the_next_one_right(vb, graph):
    """Margin ties at every point: no pass can decide them, folded or not, and the shared queue
    is too short. The call says so; the handles serve the next batch, folded as before."""
    net = synth.make_net(846, [40, 64, 64, 5], "relu", 2.0, "normal")
    D = oracle.eval_point(net, synth.make_query(846, 1, 40, 1, 0), 0)["D"]
    tied = {**net, "W": [w.copy() for w in net["W"]], "b": [b.copy() for b in net["b"]]}
    tied["W"][2][(D + 1) % 5] = tied["W"][2][D]
    tied["b"][2][(D + 1) % 5] = tied["b"][2][D]
    q = synth.make_query(846, 1, 40, 2, 20)
    n = oracle.space_size(2, 20)
    vnet = vb.Net(tied)
    res = vb.result_create_batch(vnet, 2, max_points=n, max_s=2, max_k=20, queue_cap=600)
    small = dict(q, k=8)
    for _ in range(2):
        with pytest.raises(vb.VbmcError, match="queue"):
            vb.verify_batch(vnet, res, [q, q], precision="fp32", bitmap=True, graph=graph)
        for r, s in zip(res, vb.verify_batch(vnet, res, [small, small], precision="fp32", bitmap=True, graph=graph)):
            assert s["n_recheck"][0] == 289 and s["n_recheck"][2] == 0  # folded
            compare(read(vb, r, 2, 289, tied["dims"], s), oracle.verify(tied, small), tied, small)
    for r in res:
        r.free()
    vnet.free()
